// rt_trace.cu -- persistent Monte Carlo package tracer for hierarchical grids.
//
// One CUDA thread follows one photon package at a time (Sect. 2.3): emit,
// locate the leaf, step cell by cell, lose weight by continuous absorption
// (Sect. 2.3, Lucy 1999) or by analog absorption events, scatter with the
// Henyey-Greenstein phase function, peel off scattered light towards each
// observer after every scattering (Sect. 2.4), play Russian roulette
// (Sect. 2.3), and leave at the outer boundary of the root grid.
//
// GPU design (not the paper's grid-by-grid CPU scheme, App. A):
//  * persistent grid; each warp refills its finished lanes in one batch from
//    a global package counter (one atomicAdd per refill), so warps stay full
//    while packages of very different lengths finish;
//  * the trace and the peel-off march share one cell-stepping loop: a lane
//    is either tracing or marching towards observer o, so scattering events
//    do not serialise the warp on a nested loop;
//  * geometry runs in leaf-local coordinates (cell = 1 unit, Sect. 2.3) plus
//    integer lattice coordinates at the leaf's level, so FP32 keeps its
//    precision at deep levels; a face crossing moves to the sibling in the
//    same octet (or the root-level neighbour) with one load, otherwise
//    re-descends from the root;
//  * every pass of the loop loads exactly one node word per lane: a refined
//    node advances the descent by one level, a leaf gets one segment, so a
//    lane re-descending several levels never holds up the rest of its warp;
//  * one 32-bit node word per visit (density or child index), absorbed
//    energy by FP64 atomics (RED) into [bin][cell].
#include <math_constants.h>

#include <algorithm>
#include <cfloat>
#include <type_traits>
#include <cstring>

#include "philox.cuh"
#include "rt_internal.cuh"
#include "rt_device.cuh"

namespace rtk {

// ------------------------------------------------------------------------
// shared-memory state of the tracer
// ------------------------------------------------------------------------
enum { L_EMIT = 0, L_ABS, L_ESC, L_RRG, L_RRL, L_KILL, L_PEEL, L_ND };
enum { U_PK = 0, U_CROSS, U_SCAT, U_PCROSS, U_KILL, U_POUT, U_DEFER, U_NU };
// the resampling counters (rare events) go straight to the job's ledger: two
// more per-warp counters cost the stepping loop registers

// Energy ledger per warp, updated with shared-memory atomics at package
// events (a few per package).  Two slots per warp, each tagged with the job
// it belongs to: in a batched launch a warp moves from job to job, and at
// each refill a slot that no live lane still books to is flushed to the
// job's global ledger and re-tagged to the job being emitted, so the old
// job's packages finish in one slot while the new job's start in the other.
// A lane whose job has no slot (a third job inside one warp) books directly
// to global memory.  Kept per warp rather than per thread: shared memory
// taken here is L1 cache lost to the node loads.
// Energies are kept as the bits of an FP64 sum (FP64 tracer) or as 64-bit
// fixed point, value * 2^shift of the slot's job (FP32 tracer: integer adds
// are exact, order-independent and stay off the narrow FP64 pipe).
struct WarpLedger {
  unsigned long long d[2][L_ND][8];
  unsigned long long u[2][U_NU][8];
  int tag[2][8];
  int shift[2][8];
};

// Cold per-lane state: touched at emission, scattering and peel-off
// events only, so it lives in shared memory instead of registers.
template <typename R>
struct ColdState {
  uint32_t k0[256], k1[256], c0[256], c1[256], c3[256], next[256];
  long long log_index[256], pix[256], gi[256];
  R W0[256], pw[256], gpar[256];
  int bin[256], nscat[256], obs_i[256], job[256];
  uint32_t crowd[256];  // crossings whose deposits are summed over the warp
  // scattering point and incoming direction, saved during the peel-off
  uint32_t scx[256], scy[256], scz[256], sidx[256];
  int slev[256];
  R sfx[256], sfy[256], sfz[256], sdx[256], sdy[256], sdz[256];
  // the last Philox block (four words) drawn by the lane and its index: the
  // draws of an event come from consecutive words of one block
  uint4 rblk[256];
  uint32_t rtag[256];
};

template <typename R>
__device__ __forceinline__ uint32_t draw_u32(ColdState<R>& C, int t) {
  const uint32_t j = C.next[t];
  C.next[t] = j + 1u;
  uint4 b;
  if (C.rtag[t] == (j >> 2)) {
    b = C.rblk[t];
  } else {
    b = philox4x32_10(make_uint4(C.c0[t], C.c1[t], j >> 2, C.c3[t]), C.k0[t], C.k1[t]);
    C.rblk[t] = b;
    C.rtag[t] = j >> 2;
  }
  const uint32_t w = j & 3u;
  return w == 0u ? b.x : (w == 1u ? b.y : (w == 2u ? b.z : b.w));
}

template <typename R>
__device__ __forceinline__ R draw(ColdState<R>& C, int t) {
  return Num<R>::uni(draw_u32(C, t));
}

// the ledger's sums and counts are contiguous, in the order of L_* and U_*
static_assert(offsetof(LedgerDev, peeled) == offsetof(LedgerDev, emitted) + 8 * L_PEEL, "ledger layout");
static_assert(offsetof(LedgerDev, n_peel_deferred) == offsetof(LedgerDev, n_packets) + 8 * U_DEFER, "ledger layout");
__device__ __forceinline__ double* ledger_d(LedgerDev* L, int i) { return &L->emitted + i; }
__device__ __forceinline__ unsigned long long* ledger_u(LedgerDev* L, int i) { return &L->n_packets + i; }

// floor(v * 2^shift) for v >= 0 from the bits of v, on the integer pipe
// (saturates at 2^63; zero and denormals give 0)
__device__ __forceinline__ unsigned long long to_fixed(float v, int shift) {
  const uint32_t b = __float_as_uint(v);
  const int e = (int)(b >> 23);
  const unsigned long long m = (unsigned long long)((b & 0x7FFFFFu) | 0x800000u);
  const int sh = e - 150 + shift;  // v = m * 2^(e - 150)
  const unsigned long long q =
      sh >= 0 ? (sh > 39 ? (1ull << 63) : (m << sh)) : (sh <= -24 ? 0ull : (m >> (-sh)));
  return e == 0 ? 0ull : q;
}

template <typename R>
struct SlotNum;
template <>
struct SlotNum<float> {
  static __device__ __forceinline__ void add(unsigned long long* slot, float v, int shift) {
    atomicAdd(slot, to_fixed(v, shift));
  }
  static __device__ __forceinline__ double value(unsigned long long q, int shift) { return ldexp((double)q, -shift); }
};
template <>
struct SlotNum<double> {
  static __device__ __forceinline__ void add(unsigned long long* slot, double v, int) {
    atomicAdd(reinterpret_cast<double*>(slot), v);
  }
  static __device__ __forceinline__ double value(unsigned long long q, int) { return __longlong_as_double((long long)q); }
};

// Sum of a fixed-point energy / a count over the lanes of mask m, exact: the
// value is summed in limbs narrow enough that 32 of them fit one 32-bit
// warp reduction.
__device__ __forceinline__ unsigned long long sum_lanes_u64(unsigned m, unsigned long long q) {
  const unsigned a = __reduce_add_sync(m, (unsigned)q & 0x3FFFFFu);
  const unsigned b = __reduce_add_sync(m, (unsigned)(q >> 22) & 0x3FFFFFu);
  const unsigned c = __reduce_add_sync(m, (unsigned)(q >> 44));
  return (unsigned long long)a + ((unsigned long long)b << 22) + ((unsigned long long)c << 44);
}
__device__ __forceinline__ unsigned long long sum_lanes_u32(unsigned m, uint32_t v) {
  const unsigned a = __reduce_add_sync(m, v & 0xFFFFu), b = __reduce_add_sync(m, v >> 16);
  return (unsigned long long)a + ((unsigned long long)b << 16);
}

// The slot of the job that all calling lanes (mask m) book entry i to; -1:
// they book to several jobs or entries (lanes of different call sites can
// meet where the compiler shares their code), or to a job without a slot.
__device__ __forceinline__ int common_slot(const WarpLedger& SL, unsigned m, int job, int i, int wid) {
  const int key = job * 32 + i;
  const bool same = __all_sync(m, key == __shfl_sync(m, key, __ffs(m) - 1));
  if (!same) return -1;
  return SL.tag[0][wid] == job ? 0 : (SL.tag[1][wid] == job ? 1 : -1);
}

// Bookings come in batches: the lanes that book together are summed in
// registers and one of them updates the slot.  (A 64-bit atomic add to
// shared memory is a compare-and-swap loop, which 8 to 32 lanes adding to
// one address run 8 to 32 times.)
template <typename R>
__device__ __forceinline__ void book_d(WarpLedger& SL, const JobDev* jobs, int job, int wid, int i, R v) {
  if (v == R(0)) return;
  if (sizeof(R) == 4) {
    const unsigned m = __activemask();
    const int sl = common_slot(SL, m, job, i, wid);
    if (sl >= 0) {
      const unsigned long long q = sum_lanes_u64(m, to_fixed((float)v, SL.shift[sl][wid]));
      if ((threadIdx.x & 31) == (unsigned)(__ffs(m) - 1)) atomicAdd(&SL.d[sl][i][wid], q);
      return;
    }
  }
  if (SL.tag[0][wid] == job) {
    SlotNum<R>::add(&SL.d[0][i][wid], v, SL.shift[0][wid]);
  } else if (SL.tag[1][wid] == job) {
    SlotNum<R>::add(&SL.d[1][i][wid], v, SL.shift[1][wid]);
  } else {
    atomicAdd(ledger_d(jobs[job].ledger, i), (double)v);
  }
}

__device__ __forceinline__ void book_u(WarpLedger& SL, const JobDev* jobs, int job, int wid, int i, uint32_t v) {
  if (v == 0u) return;
  const unsigned m = __activemask();
  const int sl = common_slot(SL, m, job, i, wid);
  if (sl >= 0) {
    const unsigned long long q = sum_lanes_u32(m, v);
    if ((threadIdx.x & 31) == (unsigned)(__ffs(m) - 1)) atomicAdd(&SL.u[sl][i][wid], q);
  } else if (SL.tag[0][wid] == job) {
    atomicAdd(&SL.u[0][i][wid], (unsigned long long)v);
  } else if (SL.tag[1][wid] == job) {
    atomicAdd(&SL.u[1][i][wid], (unsigned long long)v);
  } else {
    atomicAdd(ledger_u(jobs[job].ledger, i), (unsigned long long)v);
  }
}

// Warp-uniform: give job nj a ledger slot if it has none, flushing a slot
// that no live lane (lane_job: the lane's job, -1 if not live) books to.
template <typename R>
__device__ __forceinline__ void ledger_retag(WarpLedger& SL, const JobDev* jobs, int wid, int lane, int nj,
                                             int lane_job) {
  const unsigned FULL = 0xFFFFFFFFu;
  if (nj < 0 || SL.tag[0][wid] == nj || SL.tag[1][wid] == nj) return;
  const bool use0 = __any_sync(FULL, lane_job >= 0 && lane_job == SL.tag[0][wid]);
  const bool use1 = __any_sync(FULL, lane_job >= 0 && lane_job == SL.tag[1][wid]);
  const int sl = !use0 ? 0 : (!use1 ? 1 : -1);
  if (sl < 0) return;
  __syncwarp();
  const int old = SL.tag[sl][wid];
  if (old >= 0) {
    LedgerDev* L = jobs[old].ledger;
    if (lane < L_ND) {
      const unsigned long long q = SL.d[sl][lane][wid];
      if (q) atomicAdd(ledger_d(L, lane), SlotNum<R>::value(q, SL.shift[sl][wid]));
      SL.d[sl][lane][wid] = 0ull;
    } else if (lane < L_ND + U_NU) {
      const unsigned long long v = SL.u[sl][lane - L_ND][wid];
      if (v) atomicAdd(ledger_u(L, lane - L_ND), v);
      SL.u[sl][lane - L_ND][wid] = 0ull;
    }
  }
  __syncwarp();
  if (lane == 0) {
    SL.tag[sl][wid] = nj;
    SL.shift[sl][wid] = jobs[nj].led_shift;
  }
  __syncwarp();
}

template <typename R>
__device__ __forceinline__ void ledger_init(WarpLedger& SL, int wid, int lane) {
  if (lane < L_ND) SL.d[0][lane][wid] = SL.d[1][lane][wid] = 0ull;
  if (lane < U_NU) SL.u[0][lane][wid] = SL.u[1][lane][wid] = 0ull;
  if (lane < 2) SL.tag[lane][wid] = -1;
  __syncwarp();
}

template <typename R>
__device__ __forceinline__ void ledger_flush(WarpLedger& SL, const JobDev* jobs, int wid, int lane) {
  __syncwarp();
  if (lane < 2) {
    const int tag = SL.tag[lane][wid];
    if (tag >= 0) {
      LedgerDev* L = jobs[tag].ledger;
#pragma unroll
      for (int i = 0; i < L_ND; ++i)
        if (SL.d[lane][i][wid]) atomicAdd(ledger_d(L, i), SlotNum<R>::value(SL.d[lane][i][wid], SL.shift[lane][wid]));
#pragma unroll
      for (int i = 0; i < U_NU; ++i)
        if (SL.u[lane][i][wid]) atomicAdd(ledger_u(L, i), SL.u[lane][i][wid]);
    }
  }
}

enum { ST_DEAD = 0, ST_TRACE = 1, ST_PEEL = 2, ST_DONE = 3 };
enum { EV_NONE = 0, EV_IDLE, EV_INTERACT, EV_ESCAPE, EV_CUT, EV_KILL, EV_DEGEN, EV_TILE, EV_SPLIT };

// A lane that meets an event (scattering, escape, tile change, ...) waits in
// the stepping loop until `batch` lanes of its warp have one, or until no
// lane is stepping any more; the warp then leaves the loop and serves the
// waiting events together.  Each visit to the event code costs the warp the
// same whatever the number of lanes it serves, so serving one event per
// visit (batch 1) spends most issue slots on lanes that do nothing.
// The batch is the launch's: 12, and 16 for the tiled rounds and for launches
// of several jobs (small models, whose packages live for few passes).
// Batches of 8 / 10 / 12 / 16 / 20 lanes: the tiled rounds of a 256^3 cloud
// step (4e7 packages) 180.8 / 167.8 / 158.9 / 153.4 / 156.1 ms, where most
// events write a record; the untiled 128^3 cloud (4e6 packages) 5.17 / 5.08 /
// 5.11 / 5.35 / 5.76 ms, a batched launch of 16 models 8.00 / 7.80 / 7.69 /
// 7.49 / 7.80 ms.
// the marches: 8 / 12 / 16 lanes, 256^3 cloud step 138.7 / 138.5 / 135.5 ms,
// tabulated maps 3.44 / 3.34 / 3.23 ms, FP64 map 3.43 / 3.33 / 3.32 ms, deep
// cloud 6.41 / 6.54 / 6.46 ms
#ifndef RT_PEEL_EV_BATCH
#define RT_PEEL_EV_BATCH 16
#endif
// counter slot for each calling lane with one atomic per group of lanes
// that arrive together (the tile-record and peel-off queues have one
// counter each, which every lane of the device increments)
__device__ __forceinline__ unsigned long long claim_slot(unsigned long long* ctr) {
  const unsigned m = __activemask();
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  // (lanes that claim from the two queues can meet here)
  const unsigned long long c = (unsigned long long)ctr;
  if (!__all_sync(m, c == __shfl_sync(m, c, leader))) return atomicAdd(ctr, 1ull);
  unsigned long long base = 0ull;
  if (lane == leader) base = atomicAdd(ctr, (unsigned long long)__popc(m));
  base = __shfl_sync(m, base, leader);
  return base + (unsigned long long)__popc(m & ((1u << lane) - 1u));
}

// Work items for the dead lanes of a warp: the item of each lane (at or
// beyond n: none left).  A warp's first 32 items follow from its number in
// the grid, the rest come from a counter, and a warp that has seen the end
// does not ask again.  The counter is one address, its atomics take their
// turns a few ns apart: by the counter alone a launch of 1e5 packages makes
// 1.2e4 of them, most for nothing.  state (the warp's, in shared memory): 0
// nothing taken yet, 1 the end was seen, 2 the warp's own taken.  Lane 0
// stores it; a __syncwarp on either side of the store orders it against this
// and the next call's reads (shuffles and ballots bring the lanes together
// but order no memory).
__device__ __forceinline__ long long next_work(unsigned long long* counter, long long n, unsigned dead, int leader,
                                               int lane, int& state) {
  const int rank = __popc(dead & ((1u << lane) - 1u));
  const int st = state;
  __syncwarp();
  if (st == 0) {
    // (every lane is dead at a warp's first refill)
    if (lane == 0) state = 2;
    __syncwarp();
    return ((long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + rank;
  }
  if (st == 1) return n + rank;
  unsigned long long base = 0ull;
  if (lane == leader) base = atomicAdd(counter, (unsigned long long)__popc(dead));
  base = __shfl_sync(0xFFFFFFFFu, base, leader) + 32ull * gridDim.x * (blockDim.x >> 5);
  if (lane == 0 && (long long)base + __popc(dead) >= n) state = 1;
  __syncwarp();
  return (long long)base + rank;
}

// device counters of node descents (a global read of an interior cell's
// child word each: the 4 B per descent of the roofline unit), kept only in
// builds compiled with RT_COUNT_DESCENTS=1 (an atomic per descent): [0] the
// tracer's own walk, [1] peel-off marches
#ifndef RT_COUNT_DESCENTS
#define RT_COUNT_DESCENTS 0
#endif
__device__ unsigned long long g_descents[2];

// peel-off marches of warps whose live lanes all march along one axis in one
// direction run a form of the loop with the axis and direction as constants
#ifndef RT_PEEL_AXIS
#define RT_PEEL_AXIS 1
#endif

// a point source's or a beam's packages share their first cells: deposits of
// that many crossings are summed over the warp (red_acc_grouped), in a form
// of the pass of their own, which other packages do not run.  A 7e5-cell
// trace with 1.05e6 packages from a star and as many from outside: 2.25 ms
// ungrouped, 1.81 / 1.83 / 1.81 / 1.83 ms with 1 / 2 / 3 / 5 crossings; a batch
// of 16 models, half of them with a star: 7.70, 7.79 / 7.90 / 8.00 / 8.10 ms.
#ifndef RT_CROWDED
#define RT_CROWDED 1u
#endif

#ifndef RT_TRACE_ONLY_LOOP
#define RT_TRACE_ONLY_LOOP 1
#endif

__device__ __forceinline__ bool keep_stepping(int ev, int batch) {
  const unsigned waiting = __ballot_sync(0xFFFFFFFFu, ev > EV_IDLE);
  const unsigned stepping = __ballot_sync(0xFFFFFFFFu, ev == EV_NONE);
  return stepping != 0u && __popc(waiting) < batch;
}

// ------------------------------------------------------------------------
// deferred peel-off records
// ------------------------------------------------------------------------
__device__ __forceinline__ uint32_t peel_meta(int lev, int bin, int job) {
  return (uint32_t)lev | ((uint32_t)bin << 5) | ((uint32_t)job << 13);
}

template <typename R>
struct PeelIO;
template <>
struct PeelIO<float> {
  static __device__ __forceinline__ void put(void* base, unsigned long long i, const Geo<float>& g, float dx,
                                             float dy, float dz, float W, uint32_t meta) {
    uint4* p = reinterpret_cast<uint4*>(static_cast<PeelRec32*>(base) + i);
    p[0] = make_uint4(g.cx, g.cy, g.cz, g.idx);
    p[1] = make_uint4(__float_as_uint(g.fx), __float_as_uint(g.fy), __float_as_uint(g.fz), __float_as_uint(W));
    p[2] = make_uint4(__float_as_uint(dx), __float_as_uint(dy), __float_as_uint(dz), meta);
  }
  static __device__ __forceinline__ void get(const void* base, long long i, Geo<float>& g, float& dx, float& dy,
                                             float& dz, float& W, uint32_t& meta) {
    const uint4* p = reinterpret_cast<const uint4*>(static_cast<const PeelRec32*>(base) + i);
    const uint4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2);
    g.cx = a.x; g.cy = a.y; g.cz = a.z; g.idx = a.w;
    g.fx = __uint_as_float(b.x); g.fy = __uint_as_float(b.y); g.fz = __uint_as_float(b.z);
    W = __uint_as_float(b.w);
    dx = __uint_as_float(c.x); dy = __uint_as_float(c.y); dz = __uint_as_float(c.z);
    meta = c.w;
  }
};
template <>
struct PeelIO<double> {
  static __device__ __forceinline__ void put(void* base, unsigned long long i, const Geo<double>& g, double dx,
                                             double dy, double dz, double W, uint32_t meta) {
    PeelRec64* r = static_cast<PeelRec64*>(base) + i;
    *reinterpret_cast<uint4*>(&r->cx) = make_uint4(g.cx, g.cy, g.cz, g.idx);
    *reinterpret_cast<double2*>(&r->fx) = make_double2(g.fx, g.fy);
    *reinterpret_cast<double2*>(&r->fz) = make_double2(g.fz, W);
    *reinterpret_cast<double2*>(&r->dx) = make_double2(dx, dy);
    r->dz = dz;
    r->meta = meta;
  }
  static __device__ __forceinline__ void get(const void* base, long long i, Geo<double>& g, double& dx,
                                             double& dy, double& dz, double& W, uint32_t& meta) {
    const PeelRec64* r = static_cast<const PeelRec64*>(base) + i;
    const uint4 a = __ldg(reinterpret_cast<const uint4*>(&r->cx));
    const double2 b = __ldg(reinterpret_cast<const double2*>(&r->fx));
    const double2 c = __ldg(reinterpret_cast<const double2*>(&r->fz));
    const double2 d = __ldg(reinterpret_cast<const double2*>(&r->dx));
    g.cx = a.x; g.cy = a.y; g.cz = a.z; g.idx = a.w;
    g.fx = b.x; g.fy = b.y; g.fz = c.x;
    W = c.y;
    dx = d.x; dy = d.y;
    dz = __ldg(&r->dz);
    meta = __ldg(&r->meta);
  }
};
static_assert(sizeof(PeelRec32) == 48 && sizeof(PeelRec64) == 80, "peel record layout");

// Peel-off towards observer o from the scattering point g (incoming
// direction sd, weight W): the pixel the point projects to and the weight
// W p_HG(k . d_in) that reaches it before extinction (Sect. 2.4).  False
// when the point projects outside the image.
template <typename R>
__device__ __forceinline__ bool peel_setup(const JobDev& J, int o, const Geo<R>& g, R sdx, R sdy, R sdz, R W,
                                           R gpar, int bin, R& pw, long long& pix) {
  const ObsDev& O = J.obs[o];
  const R s = Num<R>::pow2m(g.lev);
  const R Px = ((R)g.cx + g.fx) * s - ObsGeom<R>::c(O, 0);
  const R Py = ((R)g.cy + g.fy) * s - ObsGeom<R>::c(O, 1);
  const R Pz = ((R)g.cz + g.fz) * s - ObsGeom<R>::c(O, 2);
  const R u = (Px * ObsGeom<R>::ex(O, 0) + Py * ObsGeom<R>::ex(O, 1) + Pz * ObsGeom<R>::ex(O, 2)) *
                  ObsGeom<R>::ip(O, 0) + R(0.5) * (R)O.nx;
  const R v = (Px * ObsGeom<R>::ey(O, 0) + Py * ObsGeom<R>::ey(O, 1) + Pz * ObsGeom<R>::ey(O, 2)) *
                  ObsGeom<R>::ip(O, 1) + R(0.5) * (R)O.ny;
  const R fu = Num<R>::floor_(u), fv = Num<R>::floor_(v);
  if (!(fu >= R(0) && fv >= R(0) && fu < (R)O.nx && fv < (R)O.ny)) return false;
  const R kx = ObsGeom<R>::k(O, 0), ky = ObsGeom<R>::k(O, 1), kz = ObsGeom<R>::k(O, 2);
  pw = W * hg_phase(gpar, sdx * kx + sdy * ky + sdz * kz);
  pix = (((long long)o * J.img_bins + (J.img_bins > 1 ? bin : 0)) * O.ny + (long long)fv) * O.nx + (long long)fu;
  return true;
}

// ------------------------------------------------------------------------
// tiled tracing: package records between rounds
// ------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ uint32_t tile_of(const Geo<R>& g, const TileRun& T) {
  const int s = g.lev + T.tsh;
  return (g.cx >> s) + (uint32_t)T.ntx * ((g.cy >> s) + (uint32_t)T.nty * (g.cz >> s));
}
// sort key of a record: (bin, tile), then the block of 2^-sbits tile edges
// the package sits in, so that a warp takes up packages that start close
// together
template <typename R>
__device__ __forceinline__ uint32_t tile_key(const Geo<R>& g, const TileRun& T, int bin) {
  const uint32_t k = (uint32_t)bin * (uint32_t)T.n_tiles + tile_of(g, T);
  if (T.sbits == 0) return k;
  const int ss = g.lev + T.tsh - T.sbits;
  const uint32_t m = (1u << T.sbits) - 1u;
  const uint32_t sub = ((g.cx >> ss) & m) | (((g.cy >> ss) & m) << T.sbits) | (((g.cz >> ss) & m) << (2 * T.sbits));
  return (k << (3 * T.sbits)) | sub;
}

// The FP32 tracer writes the narrow record unless it tracks levels or
// resamples; the FP64 record always has room for everything.
template <typename R, bool WIDE>
struct TileIO;
template <>
struct TileIO<float, false> {
  typedef TRec32 Rec;
  static __device__ __forceinline__ TRec32& b(Rec& r) { return r; }
  static __device__ __forceinline__ const TRec32& b(const Rec& r) { return r; }
  static __device__ __forceinline__ void set_ext(Rec&, uint32_t, uint32_t, uint32_t, uint32_t) {}
  static __device__ __forceinline__ void ext(const Rec&, uint32_t& o, uint32_t& s0, uint32_t& s1, uint32_t& s3) {
    o = 0xFFFFFFFFu; s0 = s1 = s3 = 0u;
  }
};
template <>
struct TileIO<float, true> {
  typedef TRec32W Rec;
  static __device__ __forceinline__ TRec32& b(Rec& r) { return r.b; }
  static __device__ __forceinline__ const TRec32& b(const Rec& r) { return r.b; }
  static __device__ __forceinline__ void set_ext(Rec& r, uint32_t o, uint32_t s0, uint32_t s1, uint32_t s3) {
    r.orig = o; r.s0 = s0; r.s1 = s1; r.s3 = s3;
  }
  static __device__ __forceinline__ void ext(const Rec& r, uint32_t& o, uint32_t& s0, uint32_t& s1, uint32_t& s3) {
    o = r.orig; s0 = r.s0; s1 = r.s1; s3 = r.s3;
  }
};
template <bool WIDE>
struct TileIO<double, WIDE> {
  typedef TRec64 Rec;
  static __device__ __forceinline__ TRec64& b(Rec& r) { return r; }
  static __device__ __forceinline__ const TRec64& b(const Rec& r) { return r; }
  static __device__ __forceinline__ void set_ext(Rec& r, uint32_t o, uint32_t s0, uint32_t s1, uint32_t s3) {
    r.orig = o; r.s0 = s0; r.s1 = s1; r.s3 = s3;
  }
  static __device__ __forceinline__ void ext(const Rec& r, uint32_t& o, uint32_t& s0, uint32_t& s1, uint32_t& s3) {
    o = r.orig; s0 = r.s0; s1 = r.s1; s3 = r.s3;
  }
};
static_assert(sizeof(TRec32) == 80 && sizeof(TRec32W) == 96 && sizeof(TRec64) == 144, "tile record layout");
__device__ __forceinline__ uint32_t pack_aux(int mlev, int plev, int sexp) {
  return (uint32_t)mlev | ((uint32_t)(plev + 1) << 8) | ((uint32_t)(sexp + 128) << 16);
}
__device__ __forceinline__ int aux_mlev(uint32_t a) { return (int)(a & 255u); }
__device__ __forceinline__ int aux_plev(uint32_t a) { return (int)((a >> 8) & 255u) - 1; }
__device__ __forceinline__ int aux_sexp(uint32_t a) { return (int)((a >> 16) & 255u) - 128; }

// N^e for the resampling factor (N^e <= 256 is checked on the host)
__device__ __forceinline__ uint32_t ipow_u(uint32_t n, int e) {
  uint32_t r = 1u;
  for (int i = 0; i < e; ++i) r *= n;
  return r;
}
// w N^-e for either sign of e
template <typename R>
__device__ __forceinline__ R scale_pow(R w, uint32_t n, int e) {
  return e >= 0 ? w / (R)ipow_u(n, e) : w * (R)ipow_u(n, -e);
}

// Subiterations: after a crossing that restarted the cursor at the root (a
// move out of the parent octet, or between root cells), the shallowest grid
// the package passed is one level below the deepest common ancestor of the
// two cells: the level of the highest lattice bit that changed on the
// crossing axis, counted from the lattice level (0 between root cells).
template <typename R>
__device__ __forceinline__ int crossed_grid_level(const Geo<R>& g, int a, R dx, R dy, R dz) {
  const uint32_t cn = a == 0 ? g.cx : (a == 1 ? g.cy : g.cz);
  const bool plus = (a == 0 ? dx : (a == 1 ? dy : dz)) > R(0);
  const uint32_t co = plus ? cn - 1u : cn + 1u;
  const int b = 31 - __clz((int)(co ^ cn));
  return g.lev > b ? g.lev - b : 0;
}

// Dust packages (Sect. 4.2): package p of an item (counted over its bins)
// is number j of the packages its cell sends in bin `bin`; the cell is the
// last one whose first package is <= the package's index within the bin.
// The package draws from the cell's own stream, counter (j + offset,
// 0x40000000 | cell), so it keeps its random numbers when the emission of
// other cells changes.  Sets the lane's stream words; returns the cell.
template <typename R>
__device__ __forceinline__ long long dust_stream(const ItemDev& I, const JobDev& J, int bin, long long p,
                                                 ColdState<R>& C, int t) {
  const long long* fb = I.dust_first + (long long)bin * (J.n_cells + 1);
  const long long kb = p - I.bin_prefix[bin];
  long long lo = 0, hi = J.n_cells - 1;
  while (lo < hi) {
    const long long mid = (lo + hi + 1) >> 1;
    if (__ldg(fb + mid) <= kb) lo = mid;
    else hi = mid - 1;
  }
  C.c0[t] = (uint32_t)(kb - __ldg(fb + lo) + J.pkt_offset);
  C.c1[t] = 0x40000000u | (uint32_t)lo;
  return lo;
}

#ifndef RT_FP32_MIN_BLOCKS
#define RT_FP32_MIN_BLOCKS 4
#endif
#ifndef RT_FP32_TILED_MIN_BLOCKS
#define RT_FP32_TILED_MIN_BLOCKS 4
#endif
// Resident blocks per SM the register allocation is sized for.  The tiled
// rounds (mode 2) run on L2-resident cells and wait on their node loads: 4
// blocks of 224 threads at 72 registers (28 warps, almost no spills) beat 3
// blocks of 256 at 80 registers (24 warps; 788 against 798 ms for the
// cloud's rounds), which beat 4 blocks of 256 at 64 registers with spills
// (861 ms); the untiled tracer keeps 4 blocks of 256.
#ifndef RT_FP32_TILED_BLOCK
#define RT_FP32_TILED_BLOCK 224
#endif
template <typename R, int MODE>
struct MinBlocks {
  static constexpr int value = sizeof(R) == 4 ? (MODE == 2 ? RT_FP32_TILED_MIN_BLOCKS : RT_FP32_MIN_BLOCKS) : 2;
};
// threads per block the tracer is compiled for (the FP32 tiled rounds may
// use fewer than 256 to fit one more block per SM)
template <typename R, int MODE>
struct MaxThreads {
  static constexpr int value = (sizeof(R) == 4 && MODE == 2) ? RT_FP32_TILED_BLOCK : 256;
};

// Whether a lane that meets a refined node goes down to its leaf within the
// pass, and takes its segment with the others, or one level per pass.  The
// first keeps more lanes at the segment, but the warp waits for the deepest
// descent: it pays where descents are frequent (the grids with a stored
// path) and short.  One level a pass / down to the leaf, each a kernel of its
// own, in ms:
//                              star's packages  dust packages  3 oblique maps
//   deep cloud, 3 levels       3.03 / 2.75 (field)             3.02 / 2.90
//   disc,  6 levels, 2.7e4     0.90 / 0.77      5.70 / 5.88    0.92 / 0.90
//   disc,  8 levels, 5.7e5     1.24 / 1.11      5.17 / 5.32    1.11 / 1.11
//   disc,  9 levels, 1.1e6     1.29 / 1.14      5.33 / 5.45    1.15 / 1.17
//   disc, 10 levels, 3.1e6     1.44 / 1.30      5.57 / 5.63    1.09 / 1.18
//   disc, 10 levels, 9.2e6     1.78 / 1.65      5.12 / 5.30    1.33 / 1.48
//   disc, 12 levels, 8.9e6     1.67 / 1.51      7.33 / 7.44    1.10 / 1.30
// The tracer gains at every depth but for dust packages, whose lives are a few
// passes; the marches lose from 10 levels on, and the line lies where they
// begin to.  (Dust packages would have the other form at any depth, a star's
// this one.)  FP64, which waits for its pipe anyway: 3.37 / 2.70 ms (32^3 clump
// with a map).  Without a stored path (128^3 cloud) 5.23 / 5.63 ms.
// A kernel of its own for each (PATH): deciding it at run time cost the
// 9.2e6-cell disc 6 %.
enum { PATH_NONE = 0, PATH_LEVEL = 1, PATH_LEAF = 2 };
template <typename R>
static int path_form(int anc) {
  return anc <= 0 ? PATH_NONE : (sizeof(R) == 8 || anc <= 8 ? PATH_LEAF : PATH_LEVEL);
}

// PATH (PATH_NONE: no): lanes keep the path above their leaf (n_anc levels) and start the
// search for a neighbour outside their octet at the deepest stored ancestor
// it shares, else at the root cell
template <typename R, bool PEEL, int EST, bool HITS, int MODE, bool LEVELS = false, bool SPLIT = false,
          int PATH = 0>
__global__ void __launch_bounds__(MaxThreads<R, MODE>::value, MinBlocks<R, MODE>::value) trace_kernel(const JobDev* __restrict__ jobs,
                                                                         const ItemDev* __restrict__ items,
                                                                         int n_items,
                                                                         unsigned long long* __restrict__ counter,
                                                                         long long total, int refill_thr,
                                                                         int ev_batch, PeelQueue Q, TileRun T,
                                                                         int n_anc) {
  typedef TileIO<R, LEVELS || SPLIT> IO;
  typedef typename IO::Rec TRec;
  const unsigned FULL = 0xFFFFFFFFu;
  __shared__ WarpLedger SL;
  __shared__ ColdState<R> C;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  __shared__ int s_work[8];  // next_work
  if (lane == 0) s_work[wid] = 0;
  ledger_init<R>(SL, wid, lane);
  C.job[t] = -1;
  C.crowd[t] = 0u;
  // per-lane state of the level-tracking and resampling tracers only: the ALI
  // emission cell of a dust package (~0u: none) and the split exponent
  // (W0 = emitted W0 / N^sexp); one element in the other tracers
  __shared__ uint32_t s_orig[(LEVELS || SPLIT) ? 256 : 1];
  __shared__ int s_sexp[SPLIT ? 256 : 1];
  uint32_t& orig_t = s_orig[(LEVELS || SPLIT) ? t : 0];
  int& sexp_t = s_sexp[SPLIT ? t : 0];
  if (LEVELS || SPLIT) orig_t = 0xFFFFFFFFu;
  // the path above the current leaf, n_anc levels per lane (dynamic shared
  // memory, n_anc x MaxThreads words)
  extern __shared__ uint32_t s_anc[];
  AncPath P;
  P.a = s_anc + t;
  P.stride = MaxThreads<R, MODE>::value;
  P.cap = PATH ? n_anc : 0;
  P.n = 0;
  __syncwarp();

  // hot per-lane state
  int st = ST_DEAD;
  Geo<R> g;
  g.cx = g.cy = g.cz = 0u;
  g.lev = 0;
  g.idx = 0u;
  g.fx = g.fy = g.fz = R(0);
  g.rho = R(0);
  Cursor cur;
  cur.pending = 0u;
  cur.k = 0;
  GridRegs G;
  G.node = nullptr;
  G.rho64 = nullptr;
  G.rx = G.ry = G.rz = 1u;
  R dx = R(0), dy = R(0), dz = R(1), ix = R(0), iy = R(0), iz = R(0);
  R W = R(0), tau = R(0), taup = R(0), pkt_abs = R(0), kext = R(0), alb = R(0), tau_cut = R(0);
  R thin_lim = R(0);       // extinction per local unit below which a deposit is taken from the f64 density
  double* absb = nullptr;
  unsigned int* hitp = nullptr;
  uint32_t step_limit = 0u, ncross = 0u, npeel = 0u;
  int mlev = 0;            // subiterations: shallowest grid level reached
  double* selfb = nullptr; // ALI: self-absorption tally (LEVELS kernels)
  int plev = -1;           // resampling: grid level of the last cell (capped), -1: none yet
  int splt_lmax = 0;       // resampling: the cap of the grid levels

  // the word (and, in FP64, the density) of the node the cursor points at
  uint32_t w = 0u;
  double r64 = 0.0;
  auto fetch_node = [&]() {
    w = ld_node(G.node + cur.pending);
    r64 = Num<R>::load_rho64(G.rho64, cur.pending);
  };

  // after a scattering (and its peel-off): new direction from the phase
  // function, Russian roulette when the weight is low, next free path.
  // Returns a fate (1 = roulette kill) or -1.
  auto finish_scatter = [&]() -> int {
    const JobDev& J = jobs[C.job[t]];
    const R mu = hg_mu(C.gpar[t], draw(C, t));
    scatter_dir(dx, dy, dz, mu, draw(C, t));
    ix = inv_abs(dx);
    iy = inv_abs(dy);
    iz = inv_abs(dz);
    const R wmin = Num<R>::rr_wmin(J);
    if (wmin > R(0) && W < wmin * C.W0[t]) {
      const R ur = draw(C, t);
      const R rp = Num<R>::rr_p(J);
      if (ur < rp) {
        book_d(SL, jobs, C.job[t], wid, L_RRL, W);
        W = R(0);
        return 1;
      }
      const R Wn = W / (R(1) - rp);
      book_d(SL, jobs, C.job[t], wid, L_RRG, Wn - W);
      W = Wn;
    }
    tau = -Num<R>::log_(draw(C, t));
    return -1;
  };

  // tiled tracing: hand the package to the next round as a record (its
  // current position, direction, weight, optical depth to the next
  // interaction, random-number position and counters)
  auto tile_push = [&]() {
    const unsigned long long slot = claim_slot(T.n_out);
    if (slot < (unsigned long long)T.cap_out) {
      TRec rr;
      auto& r = IO::b(rr);
      r.cx = g.cx; r.cy = g.cy; r.cz = g.cz;
      r.meta = peel_meta(g.lev, C.bin[t], C.job[t]);
      r.fx = g.fx; r.fy = g.fy; r.fz = g.fz; r.W = W;
      r.dx = dx; r.dy = dy; r.dz = dz; r.tau = tau;
      r.pkt_abs = pkt_abs;
      r.next = C.next[t]; r.nscat = (uint32_t)C.nscat[t]; r.ncross = ncross; r.npeel = npeel;
      r.gi = (unsigned long long)C.gi[t];
      r.aux = pack_aux(mlev, plev, SPLIT ? sexp_t : 0);
      const bool copy = SPLIT && (C.c3[t] & 0x80000000u);
      IO::set_ext(rr, orig_t, C.c0[t], C.c1[t], copy ? C.c3[t] : 0u);
      static_cast<TRec*>(T.out)[slot] = rr;
      T.out_key[slot] = tile_key(g, T, C.bin[t]);
    } else {
      atomicOr(T.status, 1);
    }
    st = ST_DEAD;
  };

  for (;;) {
    // ---------------------------------------------------------------- refill
    const unsigned dead = __ballot_sync(FULL, st == ST_DEAD);
    const unsigned busy = __ballot_sync(FULL, st == ST_TRACE || st == ST_PEEL);
    if (dead != 0u && (__popc(dead) >= refill_thr || busy == 0u)) {
      const int leader = __ffs(dead) - 1;
      const long long slot = next_work(counter, total - (MODE == 1 ? T.first : 0), dead, leader, lane, s_work[wid]);
      long long gi = MODE == 1 ? T.first + slot : slot;  // package index
      const TRec* rec = nullptr;
      if (MODE == 2 && st == ST_DEAD && slot < total) {
        rec = static_cast<const TRec*>(T.in) + slot;
        gi = (long long)IO::b(*rec).gi;
      }
      int lo = -1;
      if (st == ST_DEAD && (MODE == 2 ? rec != nullptr : gi < total)) {
        lo = 0;
        int hi = n_items - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (items[mid].pkt_begin <= gi) lo = mid;
          else hi = mid - 1;
        }
      }
      // the leader's package is the first one handed out: give its job a slot
      const int nj = __shfl_sync(FULL, lo >= 0 ? items[lo].job : -1, leader);
      ledger_retag<R>(SL, jobs, wid, lane, nj, (st == ST_TRACE || st == ST_PEEL) ? C.job[t] : -1);
      if (st == ST_DEAD) {
        if (lo < 0) {
          st = ST_DONE;
        } else if (MODE == 2) {
          // ---------------------------------- resume a package from its record
          const TRec rr = *rec;
          const auto& r = IO::b(rr);
          uint32_t x_orig, s0, s1, s3;
          IO::ext(rr, x_orig, s0, s1, s3);
          const ItemDev& I = items[lo];
          const int job = I.job;
          const JobDev& J = jobs[job];
          C.job[t] = job;
          C.gi[t] = gi;
          G.node = J.node;
          G.rho64 = J.rho64;
          G.rx = J.root[0];
          G.ry = J.root[1];
          G.rz = J.root[2];
          step_limit = (uint32_t)min(J.step_limit, (long long)0xFFFFFFFFll);
          thin_lim = sizeof(R) == 4 && J.thin64 ? R(FLT_MIN) : R(0);
          C.crowd[t] = I.kind == RT_SRC_POINT || I.kind == RT_SRC_BEAM ? RT_CROWDED : 0u;
          tau_cut = Num<R>::tau_max(J) > R(0) ? Num<R>::tau_max(J) : Num<R>::inf();
          const long long p = gi - I.pkt_begin;
          const int bin = (int)((r.meta >> 5) & 255u);
          const unsigned long long k = (unsigned long long)(p - I.bin_prefix[bin] + J.pkt_offset);
          C.bin[t] = bin;
          C.log_index[t] = J.packet_log ? I.log_offset + p : -1;
          C.k0[t] = (uint32_t)J.seed ^ J.job_id;
          C.k1[t] = (uint32_t)(J.seed >> 32) ^ J.iter;
          C.c0[t] = (uint32_t)k;
          C.c1[t] = (uint32_t)(k >> 32);
          C.c3[t] = (I.src_index << 16) | (uint32_t)bin;
          if (I.kind == RT_SRC_DUST) dust_stream(I, J, bin, p, C, t);
          if (SPLIT && (s3 & 0x80000000u)) {
            // a copy from a split: its own stream, no package log
            C.c0[t] = s0;
            C.c1[t] = s1;
            C.c3[t] = s3;
            C.log_index[t] = -1;
          }
          C.next[t] = r.next;
          C.rtag[t] = 0xFFFFFFFFu;
          const BinDev& B = J.bins[bin];
          kext = Num<R>::kext(B);
          alb = Num<R>::alb(B);
          C.gpar[t] = Num<R>::gg(B);
          if (LEVELS) {
            mlev = aux_mlev(r.aux);
            orig_t = x_orig;
            selfb = J.self_abs ? J.self_abs + (long long)bin * J.n_cells : nullptr;
          }
          absb = J.absorbed ? J.absorbed + (long long)(LEVELS ? mlev : (J.abs_bins > 1 ? bin : 0)) * J.n_cells
                            : nullptr;
          if (HITS) hitp = J.hits;
          C.W0[t] = Num<R>::w0(I, bin);
          if (SPLIT) {
            plev = aux_plev(r.aux);
            sexp_t = aux_sexp(r.aux);
            splt_lmax = J.split_lmax;
            C.W0[t] = scale_pow(C.W0[t], (uint32_t)J.split_n, sexp_t);
          }
          C.nscat[t] = (int)r.nscat;
          W = r.W;
          tau = r.tau;
          pkt_abs = r.pkt_abs;
          ncross = r.ncross;
          npeel = r.npeel;
          g.cx = r.cx; g.cy = r.cy; g.cz = r.cz;
          g.lev = (int)(r.meta & 31u);
          g.fx = r.fx; g.fy = r.fy; g.fz = r.fz;
          g.idx = 0u;
          g.rho = R(0);
          dx = r.dx; dy = r.dy; dz = r.dz;
          ix = inv_abs(dx);
          iy = inv_abs(dy);
          iz = inv_abs(dz);
          // the package sits on the face of a root cell of this tile:
          // descend from that root cell
          cur.pending = (g.cx >> g.lev) + G.rx * ((g.cy >> g.lev) + G.ry * (g.cz >> g.lev));
          cur.k = 0;
          P.n = P.cap;
          st = ST_TRACE;
          fetch_node();
        } else {
          // ------------------------------------------------ emission (Sect. 2.3)
          const ItemDev& I = items[lo];
          const int job = I.job;
          const JobDev& J = jobs[job];
          C.job[t] = job;
          C.gi[t] = gi;
          G.node = J.node;
          G.rho64 = J.rho64;
          G.rx = J.root[0];
          G.ry = J.root[1];
          G.rz = J.root[2];
          step_limit = (uint32_t)min(J.step_limit, (long long)0xFFFFFFFFll);
          thin_lim = sizeof(R) == 4 && J.thin64 ? R(FLT_MIN) : R(0);
          C.crowd[t] = I.kind == RT_SRC_POINT || I.kind == RT_SRC_BEAM ? RT_CROWDED : 0u;
          tau_cut = Num<R>::tau_max(J) > R(0) ? Num<R>::tau_max(J) : Num<R>::inf();
          const long long p = gi - I.pkt_begin;
          int blo = 0, bhi = J.n_lambda - 1;
          while (blo < bhi) {
            const int mid = (blo + bhi + 1) >> 1;
            if (I.bin_prefix[mid] <= p) blo = mid;
            else bhi = mid - 1;
          }
          const int bin = blo;
          const unsigned long long k = (unsigned long long)(p - I.bin_prefix[bin] + J.pkt_offset);
          C.bin[t] = bin;
          C.log_index[t] = J.packet_log ? I.log_offset + p : -1;
          C.k0[t] = (uint32_t)J.seed ^ J.job_id;
          C.k1[t] = (uint32_t)(J.seed >> 32) ^ J.iter;
          C.c0[t] = (uint32_t)k;
          C.c1[t] = (uint32_t)(k >> 32);
          C.c3[t] = (I.src_index << 16) | (uint32_t)bin;
          C.next[t] = 0u;
          C.rtag[t] = 0xFFFFFFFFu;
          const BinDev& B = J.bins[bin];
          kext = Num<R>::kext(B);
          alb = Num<R>::alb(B);
          C.gpar[t] = Num<R>::gg(B);
          absb = J.absorbed ? J.absorbed + (long long)(J.abs_bins > 1 ? bin : 0) * J.n_cells : nullptr;
          if (HITS) hitp = J.hits;
          const R W0 = Num<R>::w0(I, bin);
          C.W0[t] = W0;
          W = W0;
          if (SPLIT) {
            // the external field enters through the root grid (Sect. 2.2)
            plev = I.kind == RT_SRC_EXTERNAL ? 0 : -1;
            sexp_t = 0;
            splt_lmax = J.split_lmax;
          }
          pkt_abs = R(0);
          ncross = npeel = 0u;
          C.nscat[t] = 0;
          book_d(SL, jobs, job, wid, L_EMIT, W0);
          book_u(SL, jobs, job, wid, U_PK, 1u);
          bool inside;
          if (I.kind == RT_SRC_POINT || I.kind == RT_SRC_BEAM) {
            if (I.kind == RT_SRC_POINT) {
              const R u1 = draw(C, t), u2 = draw(C, t);
              iso_dir(u1, u2, dx, dy, dz);
            } else {
              dx = Num<R>::dir(I, 0);
              dy = Num<R>::dir(I, 1);
              dz = Num<R>::dir(I, 2);
            }
            inside = place_root(G, g, cur, Num<R>::pos(I, 0), Num<R>::pos(I, 1), Num<R>::pos(I, 2), dx, dy, dz);
            P.n = P.cap;
          } else if (I.kind == RT_SRC_EXTERNAL) {
            // face by area, uniform point on it, cosine-weighted inward direction
            const R ax = (R)G.ry * (R)G.rz, ay = (R)G.rx * (R)G.rz, az = (R)G.rx * (R)G.ry;
            const R v = draw(C, t) * (R(2) * (ax + ay + az));
            int face = 5;
            R cum = R(0);
            const R ar[3] = {ax, ay, az};
#pragma unroll
            for (int f = 0; f < 6; ++f) {
              cum += ar[f >> 1];
              if (face == 5 && v < cum) face = f;
            }
            const int a = face >> 1;
            const R u1 = draw(C, t), u2 = draw(C, t);
            const R u3 = draw(C, t), u4 = draw(C, t);
            const R mu = Num<R>::sqrt_(u3), st_ = Num<R>::sqrt_(fmax(R(0), R(1) - mu * mu));
            R sp, cp;
            Num<R>::sincos2pi(u4, &sp, &cp);
            const R dn = (face & 1) ? -mu : mu;
            R px, py, pz;
            if (a == 0) {
              px = (face & 1) ? (R)G.rx : R(0);
              py = u1 * (R)G.ry;
              pz = u2 * (R)G.rz;
              dx = dn; dy = st_ * cp; dz = st_ * sp;
            } else if (a == 1) {
              py = (face & 1) ? (R)G.ry : R(0);
              px = u1 * (R)G.rx;
              pz = u2 * (R)G.rz;
              dy = dn; dx = st_ * cp; dz = st_ * sp;
            } else {
              pz = (face & 1) ? (R)G.rz : R(0);
              px = u1 * (R)G.rx;
              py = u2 * (R)G.ry;
              dz = dn; dx = st_ * cp; dy = st_ * sp;
            }
            inside = place_root(G, g, cur, px, py, pz, dx, dy, dz);
            P.n = P.cap;
          } else {
            // dust emission (Sect. 4.2): the package is one of the packages
            // its cell sends in this bin, and draws from that cell's stream
            const long long clo = dust_stream(I, J, bin, p, C, t);
            const uint64_t cw = J.coord[clo];
            g.cx = (uint32_t)(cw & RT_COORD_MASK);
            g.cy = (uint32_t)((cw >> RT_COORD_BITS) & RT_COORD_MASK);
            g.cz = (uint32_t)((cw >> (2 * RT_COORD_BITS)) & RT_COORD_MASK);
            g.lev = J.level[clo];
            g.fx = draw(C, t);
            g.fy = draw(C, t);
            g.fz = draw(C, t);
            cur.pending = (uint32_t)clo;
            cur.k = g.lev;
            P.n = 0;  // placed in its leaf: no path above it yet
            const R u4 = draw(C, t), u5 = draw(C, t);
            iso_dir(u4, u5, dx, dy, dz);
            inside = true;
          }
          ix = inv_abs(dx);
          iy = inv_abs(dy);
          iz = inv_abs(dz);
          tau = -Num<R>::log_(draw(C, t));
          if (LEVELS) {
            // a package starts in the grid of its emission cell
            mlev = g.lev;
            absb = J.absorbed ? J.absorbed + (long long)mlev * J.n_cells : nullptr;
            orig_t = I.kind == RT_SRC_DUST ? cur.pending : 0xFFFFFFFFu;
            selfb = J.self_abs ? J.self_abs + (long long)bin * J.n_cells : nullptr;
            if (selfb && J.self_emit && I.kind == RT_SRC_DUST) {
              atomicAdd(J.self_emit + (long long)bin * J.n_cells + cur.pending, widen(W));
              atomicAdd(J.self_cnt + cur.pending, 1u);
            }
          }
          if (inside) {
            st = ST_TRACE;
            if (MODE != 1) fetch_node();
          } else {
            book_d(SL, jobs, job, wid, L_ESC, W);
            const long long li = C.log_index[t];
            if (li >= 0) {
              double* r = J.packet_log + li * 10;
              r[0] = (double)W; r[1] = 0.0; r[2] = 0.0; r[3] = 0.0;
              r[4] = r[5] = r[6] = 0.0;
              r[7] = (double)dx; r[8] = (double)dy; r[9] = (double)dz;
            }
            st = ST_DEAD;
          }
        }
      }
    }
    if (MODE == 1) {
      // emission round of tiled tracing: every emitted package becomes a
      // record keyed by its (bin, tile)
      if (st == ST_TRACE) tile_push();
      if (__ballot_sync(FULL, st == ST_DEAD) == 0u) break;
      continue;
    }
    if (__ballot_sync(FULL, st == ST_TRACE || st == ST_PEEL) == 0u) {
      // nothing to step: finished, or packages that left at emission
      if (__ballot_sync(FULL, st == ST_DEAD) == 0u) break;
      continue;
    }

    // ------------------------------------------------------------- fast path
    // Step cells until ev_batch lanes of the warp have met an event, or
    // none steps any more.  A leaf gets one segment (Sect. 2.3) and a face
    // crossing; a refined node advances the descent by a level, which takes
    // the lane's pass, or down to the leaf within the pass (PATH_LEAF).  The
    // word of the next node is fetched as soon as the crossing has named it,
    // so the segment's absorption and deposit run while the load is under way.
    int ev = (st == ST_TRACE || st == ST_PEEL) ? EV_NONE : EV_IDLE;
    // one pass of the loop; a warp none of whose lanes marches an inline
    // peel-off (the deferred queue had room) runs the tracing-only form
    auto pass = [&]() {
      if (ev == EV_NONE) {
        if (w & RT_INTERIOR) {
          descend_step(g, cur, w, dx, dy, dz, P);
          if (RT_COUNT_DESCENTS) atomicAdd(&g_descents[st == ST_TRACE ? 0 : 1], 1ull);
          fetch_node();
        } else {
          settle_leaf(g, cur, w, r64);
          const bool tr = st == ST_TRACE;
          const uint32_t leaf = cur.pending;
          const Exit<R> E = exit_face(g, dx, dy, dz, ix, iy, iz);
          const R tx = E.t;
          int lvs = 0;
          if (SPLIT && tr) {
            lvs = min(g.lev, splt_lmax);
            if (plev < 0) plev = lvs;
          }
          if (tr && ncross >= step_limit) {
            ev = EV_KILL;
          } else if (!Num<R>::finite(tx)) {
            ev = EV_DEGEN;  // cannot happen for |d| = 1
          } else if (SPLIT && tr && lvs != plev) {
            ev = EV_SPLIT;  // entered a grid of another level: resample first
          } else {
            const int lev = g.lev;
            const R kl = Num<R>::down(kext * g.rho, lev);  // extinction per local unit
            // continuous: the free path is drawn in scattering optical depth
            // (the weight decays by the absorbed fraction along the segment);
            // analog: in extinction optical depth
            const R kev = EST == RT_EST_CONTINUOUS ? alb * kl : kl;
            const R tev = kev * tx;
            const bool inside_event = tr && kev > R(0) && tev >= tau;
            R tseg = tx;
            double* const dep_to = absb;
            if (!tr) {
              taup += kl * tx;
              npeel += Num<R>::pos(tx) ? 1u : 0u;
            }
            if (inside_event) {
              tseg = tau / kev;
              g.fx = Num<R>::moved01(g.fx, tseg, dx);
              g.fy = Num<R>::moved01(g.fy, tseg, dy);
              g.fz = Num<R>::moved01(g.fz, tseg, dz);
              ev = EV_INTERACT;
            } else if (!tr && taup > tau_cut) {
              ev = EV_CUT;
            } else {
              uint32_t moved;
              const int ax = E.x ? 0 : (E.y ? 1 : 2);
              if (!cross_face(G, g, cur, leaf, E, tx, true, dx, dy, dz, moved, P)) {
                ev = EV_ESCAPE;
              } else {
                fetch_node();
                if (MODE == 2 && tr && (moved >> (lev + T.tsh)) != 0u) ev = EV_TILE;  // entered another tile: next round
                // (the search for the neighbour starts at or above the level
                // of the crossed face: cur.k <= that level)
                if (LEVELS && tr && cur.k < mlev && crossed_grid_level(g, ax, dx, dy, dz) < mlev) {
                  const JobDev& J = jobs[C.job[t]];
                  const int v = crossed_grid_level(g, ax, dx, dy, dz);
                  if (v <= J.sub_conf) {
                    ev = EV_ESCAPE;  // left the subtree of this subiteration
                  } else {
                    mlev = v;
                    absb = J.absorbed ? J.absorbed + (long long)mlev * J.n_cells : nullptr;
                  }
                }
              }
            }
            if (tr) {
              if (EST == RT_EST_CONTINUOUS) {
                R q, e;
                Num<R>::absorb_pair((kl - kev) * tseg, q, e);
                tau = inside_event ? R(0) : tau - tev;
                const R dep = W * q;
                W = W * e;
                const bool thin = sizeof(R) == 4 && !(kl >= R(FLT_MIN));
                if (dep > R(0) && !thin) {
                  pkt_abs += dep;
                  if (dep_to) red_acc(dep_to + leaf, widen(dep));
                  if (HITS && hitp) atomicAdd(hitp + leaf, 1u);
                  if (LEVELS && selfb && leaf == orig_t) atomicAdd(selfb + leaf, widen(dep));
                } else if (thin && tseg > R(0) && jobs[C.job[t]].thin64) {
                  // a near-vacuum cell: its extinction per unit length is
                  // below the f32 normal range, so the deposit is taken
                  // from the f64 density in the thin limit q = x (x <
                  // 1e-38; the weight and the free path do not change)
                  const JobDev& J = jobs[C.job[t]];
                  const BinDev& B = J.bins[C.bin[t]];
                  const double x = (1.0 - B.albedo_d) * B.kext_d * __ldg(J.rho64 + leaf) * Num<double>::pow2m(lev) *
                                   (double)tseg;
                  const double d64 = widen(W) * x;
                  if (d64 > 0.0) {
                    if (dep_to) red_acc(dep_to + leaf, d64);
                    if (HITS && hitp) atomicAdd(hitp + leaf, 1u);
                    if (LEVELS && selfb && leaf == orig_t) atomicAdd(selfb + leaf, d64);
                  }
                }
              } else {
                tau = inside_event ? R(0) : tau - tev;
              }
              ncross += tseg > R(0) ? 1u : 0u;
            }
          }
        }
      }
    };
    constexpr bool to_leaf = PATH == PATH_LEAF;
    // The tracing-only pass.  On large grids it is bound by the SM's random
    // accesses: one 4-byte load and one FP64 reduction per crossing to cells
    // in the L2 run at 1.2e11 per second at most (a kernel that does nothing
    // else; 2.9e11 loads or 2.0e11 reductions alone), and the untiled 128^3
    // cloud reaches 1.15e11.  On grids of 1e5..1e6 cells it is bound by the
    // length of its dependent chain, so everything a common segment needs is
    // straight-line; what few lanes need (a refined node, a leaf coarser than
    // the lattice level, the step limit) takes the pass for itself, and one
    // more branch holds what few segments need (an interaction inside the
    // segment, a thick segment's exponential, a near-vacuum deposit).  The
    // crossing comes before the segment's deposit, so that the word of the
    // next node is under way meanwhile (7e5 cells, 2.1e6 packages: 2.42 ms ->
    // 2.24 ms; the deposit first: 2.31 ms; fetching a whole pass ahead, with
    // the registers that takes: 2.44 to 2.55 ms).
    auto pass_trace = [&](auto grouped) {
      constexpr bool GROUPED = decltype(grouped)::value;
      if (ev != EV_NONE) return;
      if ((w & RT_INTERIOR) || cur.k < g.lev || ncross >= step_limit) {
        if (w & RT_INTERIOR) {
          do {
            descend_step(g, cur, w, dx, dy, dz, P);
            if (RT_COUNT_DESCENTS) atomicAdd(&g_descents[0], 1ull);
            fetch_node();
          } while (to_leaf && (w & RT_INTERIOR));
          if (!to_leaf) return;
        }
        if (cur.k < g.lev) settle_leaf(g, cur, w, r64);
        if (ncross >= step_limit) ev = EV_KILL;
        if (!to_leaf || ev != EV_NONE) return;
      }
      const uint32_t leaf = cur.pending;
      const int lev = g.lev;
      if (SPLIT) {
        const int lvs = min(lev, splt_lmax);
        if (plev < 0) plev = lvs;
        if (lvs != plev) {
          ev = EV_SPLIT;  // entered a grid of another level: resample first
          return;
        }
      }
      const Exit<R> E = exit_face(g, dx, dy, dz, ix, iy, iz);
      const R kl = Num<R>::down(kext * Num<R>::leaf_rho(w, r64), lev);  // extinction per local unit
      // continuous: the free path is drawn in scattering optical depth (the
      // weight decays by the absorbed fraction along the segment); analog:
      // in extinction optical depth.  tau > 0, so an interaction has kev > 0
      const R kev = EST == RT_EST_CONTINUOUS ? alb * kl : kl;
      const R tev = kev * E.t;
      const bool hit = Num<R>::ge(tev, tau);
      double* const dep_to = absb;
      R tseg = E.t, x = R(0), ex = R(1);
      if (EST == RT_EST_CONTINUOUS) {
        const R ka = kl - kev;
        x = ka * tseg;
        const bool thin = sizeof(R) == 4 && !(kl >= thin_lim);
        if (hit || !Num<R>::thin_seg(x) || thin) {
          if (hit) {
            tseg = tau / kev;
            x = ka * tseg;
          }
          if (!Num<R>::thin_seg(x)) ex = Num<R>::exp_(-x);
          if (thin && tseg > R(0)) {
            // a near-vacuum cell: its extinction per unit length is below
            // the f32 normal range, so the deposit is taken from the f64
            // density in the thin limit q = x (x < 1e-38; the weight and
            // the free path do not change)
            const JobDev& J = jobs[C.job[t]];
            const BinDev& B = J.bins[C.bin[t]];
            const double x64 = (1.0 - B.albedo_d) * B.kext_d * __ldg(J.rho64 + leaf) * Num<double>::pow2m(lev) *
                               (double)tseg;
            const double d64 = widen(W) * x64;
            if (d64 > 0.0) {
              if (dep_to) red_acc(dep_to + leaf, d64);
              if (HITS && hitp) atomicAdd(hitp + leaf, 1u);
              if (LEVELS && selfb && leaf == orig_t) atomicAdd(selfb + leaf, d64);
            }
          }
        }
      } else if (hit) {
        tseg = tau / kev;
      }
      uint32_t moved;
      const bool inside = cross_face(G, g, cur, leaf, E, tseg, !hit, dx, dy, dz, moved, P);
      ev = hit ? EV_INTERACT : (inside ? EV_NONE : EV_ESCAPE);
      if (!Num<R>::finite(E.t)) ev = EV_DEGEN;  // cannot happen for |d| = 1
      if (ev == EV_NONE) {
        fetch_node();
        if (MODE == 2 && (moved >> (lev + T.tsh)) != 0u) ev = EV_TILE;  // entered another tile: next round
        // (the search for the neighbour starts at or above the level of the
        // crossed face: cur.k <= that level)
        if (LEVELS && cur.k < mlev) {
          const int v = crossed_grid_level(g, E.x ? 0 : (E.y ? 1 : 2), dx, dy, dz);
          if (v < mlev) {
            const JobDev& J = jobs[C.job[t]];
            if (v <= J.sub_conf) {
              ev = EV_ESCAPE;  // left the subtree of this subiteration
            } else {
              mlev = v;
              absb = J.absorbed ? J.absorbed + (long long)mlev * J.n_cells : nullptr;
            }
          }
        }
      }
      if (EST == RT_EST_CONTINUOUS) {
        R q, e;
        Num<R>::absorb_given(x, ex, q, e);
        const R dep = W * q;
        W = W * e;
        if (Num<R>::pos(dep) && (sizeof(R) != 4 || kl >= R(FLT_MIN))) {
          pkt_abs += dep;
          if (GROUPED && ncross < C.crowd[t]) {
            if (dep_to || (HITS && hitp))
              red_acc_grouped(dep_to ? dep_to + leaf : nullptr, HITS && hitp ? hitp + leaf : nullptr, widen(dep));
          } else {
            if (dep_to) red_acc(dep_to + leaf, widen(dep));
            if (HITS && hitp) atomicAdd(hitp + leaf, 1u);
          }
          if (LEVELS && selfb && leaf == orig_t) atomicAdd(selfb + leaf, widen(dep));
        }
      }
      tau = hit ? R(0) : tau - tev;
      ncross += Num<R>::pos(tseg) ? 1u : 0u;
    };
    // every lane that leaves EV_NONE in the loop waits with an event
    const int stay = max(0, __popc(__ballot_sync(FULL, ev == EV_NONE)) - ev_batch);
    if (RT_TRACE_ONLY_LOOP && (!PEEL || __ballot_sync(FULL, st == ST_PEEL) == 0u)) {
      // packages fresh from a point source or a beam
      for (int i = 0; i < 64 && __any_sync(FULL, ev == EV_NONE && ncross < C.crowd[t]); ++i)
        pass_trace(std::true_type{});
      do {
        pass_trace(std::false_type{});
      } while (__popc(__ballot_sync(FULL, ev == EV_NONE)) > stay);
    } else {
      do {
        pass();
      } while (__popc(__ballot_sync(FULL, ev == EV_NONE)) > stay);
    }

    // ------------------------------------------------------------- slow path
    if (ev == EV_NONE || ev == EV_IDLE) continue;
    int fate = -1;  // >= 0: the package ends with this fate
    bool pick_observer = false;
    const int job = C.job[t];
    if (ev == EV_KILL || (ev == EV_DEGEN && st == ST_TRACE)) {
      book_d(SL, jobs, job, wid, L_KILL, W);
      book_u(SL, jobs, job, wid, U_KILL, 1u);
      atomicOr(&jobs[job].ledger->status, ev == EV_KILL ? 1 : 2);
      fate = 2;
    } else if (ev == EV_DEGEN || ev == EV_CUT) {
      pick_observer = true;  // abandon this observer
    } else if (ev == EV_ESCAPE) {
      if (st == ST_TRACE) {
        book_d(SL, jobs, job, wid, L_ESC, W);
        fate = 0;
      } else {
        // the peel-off contribution reaches the observer (Sect. 2.4)
        const R c = C.pw[t] * Num<R>::exp_(-taup);
        if (c > R(0)) atomicAdd(jobs[job].images + C.pix[t], widen(c));
        book_d(SL, jobs, job, wid, L_PEEL, c);
        pick_observer = true;
      }
    } else if (MODE == 2 && ev == EV_TILE) {
      tile_push();
    } else if (SPLIT && ev == EV_SPLIT) {
      // Resampling at a grid boundary (Sect. 2.3).  Entering a grid dl
      // levels deeper: M = N^dl packages of weight W/M at this point and
      // direction; the copies are written as records for the next round,
      // each with the stream named by three words drawn here and the copy
      // index, and a free path from that stream.  Leaving for a grid dl
      // levels shallower: survive with probability 1/M (integer test on one
      // word), carrying M W.  W0 follows the weight.
      const JobDev& J = jobs[job];
      const int lv = min(g.lev, splt_lmax);
      const int dl = lv - plev;
      plev = lv;
      if (dl > 0) {
        const uint32_t M = ipow_u((uint32_t)J.split_n, dl);
        const uint32_t w0 = draw_u32(C, t), w1 = draw_u32(C, t), w2 = draw_u32(C, t);
        const unsigned long long need = (unsigned long long)(M - 1u);
        const unsigned long long base = atomicAdd(T.n_split, need);
        if (base + need <= (unsigned long long)T.split_cap) {
          W = W / (R)M;
          C.W0[t] = C.W0[t] / (R)M;
          sexp_t += dl;
          const unsigned long long slot0 = atomicAdd(T.n_out, need);
          const uint32_t key = tile_key(g, T, C.bin[t]);
          for (uint32_t kk = 1u; kk < M; ++kk) {
            const unsigned long long slot = slot0 + kk - 1u;
            if (slot >= (unsigned long long)T.cap_out) {
              atomicOr(T.status, 1);
              break;
            }
            const uint32_t s3 = 0x80000000u | (w2 & 0x7FFFFF00u) | kk;
            const uint4 blk = philox4x32_10(make_uint4(w0, w1, 0u, s3), C.k0[t], C.k1[t]);
            TRec rr;
            auto& r = IO::b(rr);
            r.cx = g.cx; r.cy = g.cy; r.cz = g.cz;
            r.meta = peel_meta(g.lev, C.bin[t], job);
            r.fx = g.fx; r.fy = g.fy; r.fz = g.fz; r.W = W;
            r.dx = dx; r.dy = dy; r.dz = dz;
            r.tau = -Num<R>::log_(Num<R>::uni(blk.x));
            r.pkt_abs = R(0);
            r.next = 1u; r.nscat = 0u; r.ncross = 0u; r.npeel = 0u;
            r.gi = (unsigned long long)C.gi[t];
            r.aux = pack_aux(mlev, lv, sexp_t);
            IO::set_ext(rr, orig_t, w0, w1, s3);
            static_cast<TRec*>(T.out)[slot] = rr;
            T.out_key[slot] = key;
          }
          atomicAdd(&J.ledger->n_split, need);
        } else {
          atomicAdd(&J.ledger->n_split_skipped, 1ull);  // no room: the package goes on whole
        }
      } else {
        const uint32_t M = ipow_u((uint32_t)J.split_n, -dl);
        const uint32_t u = draw_u32(C, t);
        if ((unsigned long long)u * M < (1ull << 32)) {
          const R Wn = W * (R)M;
          book_d(SL, jobs, job, wid, L_RRG, Wn - W);
          W = Wn;
          C.W0[t] = C.W0[t] * (R)M;
          sexp_t += dl;
        } else {
          book_d(SL, jobs, job, wid, L_RRL, W);
          W = R(0);
          fate = 1;
        }
      }
    } else {  // EV_INTERACT: absorption (analog) or scattering in this cell
      bool scatter = true;
      if (EST == RT_EST_ANALOG) {
        const R ua = draw(C, t);
        if (ua >= alb) {
          scatter = false;
          if (absb) atomicAdd(absb + cur.pending, widen(W));
          pkt_abs += W;
          W = R(0);
          fate = 3;
        }
      }
      if (scatter) {
        C.nscat[t] += 1;
        g.idx = cur.pending;
        bool inline_peel = PEEL && jobs[job].n_obs > 0;
        if (inline_peel && Q.cap > 0) {
          // defer: the peel-off kernel marches this record to every observer
          const unsigned long long slot = claim_slot(Q.count);
          if (slot < (unsigned long long)Q.cap) {
            PeelIO<R>::put(Q.rec, slot, g, dx, dy, dz, W, peel_meta(g.lev, C.bin[t], job));
            book_u(SL, jobs, job, wid, U_DEFER, 1u);
            inline_peel = false;
          }
        }
        if (inline_peel) {
          // queue full (or none): save the scattering point and march
          // towards each observer in turn; the new direction is drawn after
          // the last observer
          C.scx[t] = g.cx; C.scy[t] = g.cy; C.scz[t] = g.cz;
          C.sidx[t] = g.idx; C.slev[t] = g.lev;
          C.sfx[t] = g.fx; C.sfy[t] = g.fy; C.sfz[t] = g.fz;
          C.sdx[t] = dx; C.sdy[t] = dy; C.sdz[t] = dz;
          C.obs_i[t] = -1;
          st = ST_PEEL;
          pick_observer = true;
        } else {
          fate = finish_scatter();
        }
      }
    }

    // -------------------------------------------- peel-off observer selection
    if (PEEL && pick_observer) {
      const JobDev& J = jobs[C.job[t]];
      // back to the scattering point
      g.cx = C.scx[t]; g.cy = C.scy[t]; g.cz = C.scz[t];
      g.idx = C.sidx[t]; g.lev = C.slev[t];
      g.fx = C.sfx[t]; g.fy = C.sfy[t]; g.fz = C.sfz[t];
      cur.pending = g.idx;
      cur.k = g.lev;
      fetch_node();
      P.n = 0;  // the stored path may be an inline peel-off march's
      const R sdx = C.sdx[t], sdy = C.sdy[t], sdz = C.sdz[t];
      int o = C.obs_i[t];
      bool started = false;
      while (!started) {
        ++o;
        if (o >= J.n_obs) break;
        R pw;
        long long pix;
        if (!peel_setup<R>(J, o, g, sdx, sdy, sdz, W, C.gpar[t], C.bin[t], pw, pix)) {
          book_u(SL, jobs, C.job[t], wid, U_POUT, 1u);
          continue;
        }
        C.pw[t] = pw;
        C.pix[t] = pix;
        const ObsDev& O = J.obs[o];
        dx = ObsGeom<R>::k(O, 0); dy = ObsGeom<R>::k(O, 1); dz = ObsGeom<R>::k(O, 2);
        ix = inv_abs(dx); iy = inv_abs(dy); iz = inv_abs(dz);
        taup = R(0);
        started = true;
      }
      C.obs_i[t] = o;
      if (!started) {
        // all observers done: continue the package from the scattering point
        dx = sdx; dy = sdy; dz = sdz;
        st = ST_TRACE;
        fate = finish_scatter();
      }
    }

    if (fate >= 0) {
      const int job = C.job[t];
      book_d(SL, jobs, job, wid, L_ABS, pkt_abs);
      book_u(SL, jobs, job, wid, U_CROSS, ncross);
      book_u(SL, jobs, job, wid, U_SCAT, (uint32_t)C.nscat[t]);
      book_u(SL, jobs, job, wid, U_PCROSS, npeel);
      const long long li = C.log_index[t];
      if (li >= 0) {
        double* r = jobs[job].packet_log + li * 10;
        const double s = (double)Num<R>::pow2m(g.lev) * jobs[job].h0;
        r[0] = fate == 0 ? (double)W : 0.0;
        r[1] = (double)C.nscat[t];
        r[2] = (double)ncross;
        r[3] = (double)fate;
        // signed lattice coordinates: a package that left through a lower
        // face sits at index -1 with offset 1
        r[4] = ((double)(int)g.cx + (double)g.fx) * s;
        r[5] = ((double)(int)g.cy + (double)g.fy) * s;
        r[6] = ((double)(int)g.cz + (double)g.fz) * s;
        r[7] = (double)dx; r[8] = (double)dy; r[9] = (double)dz;
      }
      st = ST_DEAD;
    }
  }

  // ------------------------------------------------------------ final ledger
  ledger_flush<R>(SL, jobs, wid, lane);
}

// ------------------------------------------------------------------------
// deferred peel-off (Sect. 2.4): one work item per (record, observer); each
// lane marches from the scattering point to the grid edge along k_o, summing
// the extinction optical depth, and adds W p_HG e^{-tau} to its pixel.
// Persistent warps refill finished lanes from a global counter.
// ------------------------------------------------------------------------
// Blocks per SM: 5 (48 registers), with the stored path 4 (64: the deep cloud
// 6.16 against 6.41 ms, the 256^3 cloud without it 140.3 against 138.8 ms)
#ifndef RT_PEEL_MIN_BLOCKS
#define RT_PEEL_MIN_BLOCKS 5
#endif
// work item gi = (record, observer): observer-major (neighbouring lanes
// march in the same direction from consecutive records; 237 against 257 ms
// for the cloud's six axis maps record-major)
#ifndef RT_PEEL_OBS_MAJOR
#define RT_PEEL_OBS_MAJOR 1
#endif
template <typename R, int PATH>
struct PeelMinBlocks {
  static constexpr int value = sizeof(R) == 4 ? RT_PEEL_MIN_BLOCKS - (PATH ? 1 : 0) : 2;
};

template <typename R, bool TAB, int PATH = 0>
__global__ void __launch_bounds__(256, PeelMinBlocks<R, PATH>::value) peel_kernel(const JobDev* __restrict__ jobs,
                                                                           PeelQueue Q,
                                                                           unsigned long long* __restrict__ work,
                                                                           int n_obs_max, int refill_thr,
                                                                           int n_anc) {
  const unsigned FULL = 0xFFFFFFFFu;
  enum { P_DEAD = 0, P_LIVE = 1, P_DONE = 2 };
  __shared__ WarpLedger SL;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  __shared__ int s_work[8];  // next_work
  if (lane == 0) s_work[wid] = 0;
  ledger_init<R>(SL, wid, lane);
  // the path above the current leaf (dynamic shared memory, n_anc x 256 words)
  extern __shared__ uint32_t s_anc[];
  AncPath P;
  P.a = s_anc + t;
  P.stride = 256;
  P.cap = PATH ? n_anc : 0;
  P.n = 0;
  const long long n_rec = min((long long)*Q.count, Q.cap);
  const long long total = n_rec * (long long)n_obs_max;

  // per lane: the work item (record, observer); the march direction, the
  // record's weighted phase function and its pixel are derived again where
  // needed instead of held (registers: the kernel runs 5 blocks per SM)
  int st = P_DEAD, job = -1, obs_o = 0;
  uint32_t rec_i = 0u;
  Geo<R> g;
  Cursor cur;
  GridRegs G;
  R kext = R(0), taup = R(0), tau_cut = R(0);
  uint32_t npeel = 0u;
  // accelerated peel-off: block of the scattering point (x | y << 10 | z << 20),
  // kappa_ext h0 of the bin
  uint32_t tab_blk = 0u;
  R ktab = R(0);
  // an observer along a coordinate axis (the paper's maps, Sect. 4.1): the
  // march moves on that axis only; akey = 2 x axis + (direction > 0), else -1
  int akey = -1;
  g.lev = 0;
  cur.pending = 0u;
  cur.k = 0;
  G.node = nullptr;
  G.rho64 = nullptr;
  G.rx = G.ry = G.rz = 1u;

  for (;;) {
    // ---------------------------------------------------------------- refill
    const unsigned dead = __ballot_sync(FULL, st == P_DEAD);
    const unsigned live = __ballot_sync(FULL, st == P_LIVE);
    if (dead != 0u && (__popc(dead) >= refill_thr || live == 0u)) {
      const int leader = __ffs(dead) - 1;
      const long long gi = next_work(work, total, dead, leader, lane, s_work[wid]);
      const bool have = st == P_DEAD && gi < total;
      if (st == P_DEAD && !have) st = P_DONE;
      Geo<R> rg;
      R sdx = R(0), sdy = R(0), sdz = R(0), W = R(0);
      uint32_t meta = 0u;
      int o = 0, rjob = -1;
      long long rec = 0;
      if (have) {
#if RT_PEEL_OBS_MAJOR
        rec = gi % n_rec;
        o = (int)(gi / n_rec);
#else
        rec = gi / n_obs_max;
        o = (int)(gi - rec * n_obs_max);
#endif
        PeelIO<R>::get(Q.rec, rec, rg, sdx, sdy, sdz, W, meta);
        rjob = (int)(meta >> 13);
      }
      const int nj = __shfl_sync(FULL, rjob, leader);
      ledger_retag<R>(SL, jobs, wid, lane, nj, st == P_LIVE ? job : -1);
      if (have) {
        const JobDev& J = jobs[rjob];
        if (o < J.n_obs) {
          rg.lev = (int)(meta & 31u);
          const int bin = (int)((meta >> 5) & 255u);
          const BinDev& B = J.bins[bin];
          R pw;
          long long pix;
          if (peel_setup<R>(J, o, rg, sdx, sdy, sdz, W, Num<R>::gg(B), bin, pw, pix)) {
            const ObsDev& O = J.obs[o];
            const R kx = ObsGeom<R>::k(O, 0), ky = ObsGeom<R>::k(O, 1), kz = ObsGeom<R>::k(O, 2);
            const int pax = TAB ? -1
                                : ((ky == R(0) && kz == R(0)) ? 0
                                                               : ((kx == R(0) && kz == R(0)) ? 1
                                                                                             : ((kx == R(0) && ky == R(0)) ? 2 : -1)));
            akey = pax < 0 ? -1 : 2 * pax + ((pax == 0 ? kx : (pax == 1 ? ky : kz)) > R(0) ? 1 : 0);
            obs_o = o;
            rec_i = (uint32_t)rec;
            g = rg;
            cur.pending = g.idx;
            cur.k = g.lev;
            P.n = 0;  // starts in its leaf: no path above it yet
            G.node = J.node;
            G.rho64 = J.rho64;
            G.rx = J.root[0];
            G.ry = J.root[1];
            G.rz = J.root[2];
            kext = Num<R>::kext(B);
            tau_cut = Num<R>::tau_max(J) > R(0) ? Num<R>::tau_max(J) : Num<R>::inf();
            taup = R(0);
            npeel = 0u;
            job = rjob;
            if (TAB) {
              const int sh = g.lev + J.ptab_bsh;
              tab_blk = (g.cx >> sh) | ((g.cy >> sh) << 10) | ((g.cz >> sh) << 20);
              ktab = (R)B.kext_d;
            }
            st = P_LIVE;
          } else {
            book_u(SL, jobs, rjob, wid, U_POUT, 1u);
          }
        }
      }
    }
    if (__ballot_sync(FULL, st == P_LIVE) == 0u) {
      if (__ballot_sync(FULL, st == P_DEAD) == 0u) break;
      continue;
    }

    // ----------------------------------------------------------------- march
    int ev = st == P_LIVE ? EV_NONE : EV_IDLE;
    constexpr bool to_leaf = PATH == PATH_LEAF;
    // one pass per lane and iteration.  AX >= 0: every live lane of the warp
    // marches along axis AX in direction PL (an axis observer; the work items
    // are observer-major, so this is the common case) and the axis and the
    // direction are constants; AX = -1: any direction
    auto march = [&](auto ax_c, auto pl_c) {
      constexpr int AX = decltype(ax_c)::value;
      constexpr bool PL = decltype(pl_c)::value;
      const R KA = PL ? R(1) : R(-1);
      // any direction: the observer's, from the job table
      R dx = R(0), dy = R(0), dz = R(1), ix = R(0), iy = R(0), iz = R(1);
      int pax = -1;
      bool pplus = false;
      if (AX < 0 && st == P_LIVE) {
        const ObsDev& O = jobs[job].obs[obs_o];
        dx = ObsGeom<R>::k(O, 0);
        dy = ObsGeom<R>::k(O, 1);
        dz = ObsGeom<R>::k(O, 2);
        ix = inv_abs(dx);
        iy = inv_abs(dy);
        iz = inv_abs(dz);
        pax = akey >> 1;
        pplus = (akey & 1) != 0;
      }
      do {
        if (ev == EV_NONE) {
          uint32_t w = ld_node(G.node + cur.pending);
          double r64 = Num<R>::load_rho64(G.rho64, cur.pending);
          while (to_leaf && (w & RT_INTERIOR)) {
            if (AX >= 0)
              descend_step(g, cur, w, AX == 0 ? KA : R(0), AX == 1 ? KA : R(0), AX == 2 ? KA : R(0), P);
            else
              descend_step(g, cur, w, dx, dy, dz, P);
            if (RT_COUNT_DESCENTS) atomicAdd(&g_descents[1], 1ull);
            w = ld_node(G.node + cur.pending);
            r64 = Num<R>::load_rho64(G.rho64, cur.pending);
          }
          if (w & RT_INTERIOR) {
            if (AX >= 0)
              descend_step(g, cur, w, AX == 0 ? KA : R(0), AX == 1 ? KA : R(0), AX == 2 ? KA : R(0), P);
            else
              descend_step(g, cur, w, dx, dy, dz, P);
            if (RT_COUNT_DESCENTS) atomicAdd(&g_descents[1], 1ull);
          } else {
            settle_leaf(g, cur, w, r64);
            int a;
            R tx;
            Exit<R> E;
            if (AX >= 0) {
              const R f = AX == 0 ? g.fx : (AX == 1 ? g.fy : g.fz);
              tx = PL ? R(1) - f : f;
              a = AX;
            } else if (pax >= 0) {
              // along an axis: the exit distance is the offset to the face ahead
              const R f = pax == 0 ? g.fx : (pax == 1 ? g.fy : g.fz);
              tx = pplus ? R(1) - f : f;
              a = pax;
            } else {
              E = exit_face(g, dx, dy, dz, ix, iy, iz);
              tx = E.t;
              a = E.x ? 0 : (E.y ? 1 : 2);
            }
            uint32_t moved;
            if (AX < 0 && !Num<R>::finite(tx)) {
              ev = EV_CUT;  // cannot happen for |k| = 1
            } else {
              taup += Num<R>::down(kext * g.rho, g.lev) * tx;
              npeel += Num<R>::pos(tx) ? 1u : 0u;
              if (!Num<R>::ge(tau_cut, taup)) {
                ev = EV_CUT;
              } else if (!(AX >= 0     ? advance_axis(G, g, cur, AX, PL, P)
                           : pax >= 0 ? advance_axis(G, g, cur, a, pplus, P)
                                      : cross_face(G, g, cur, g.idx, E, tx, true, dx, dy, dz, moved, P))) {
                ev = EV_ESCAPE;
              } else if (TAB && cur.k == 0) {
                const JobDev& J = jobs[job];
                const int sh = g.lev + J.ptab_bsh;
                const uint32_t bx = g.cx >> sh, by = g.cy >> sh, bz = g.cz >> sh;
                if ((bx | (by << 10) | (bz << 20)) != tab_blk) {
                  // left the scattering point's block through the face on
                  // axis a: add the tabulated column of the tile it crossed
                  const uint32_t cu = a == 0 ? g.cy : (a == 1 ? g.cz : g.cx);
                  const uint32_t cv = a == 0 ? g.cz : (a == 1 ? g.cx : g.cy);
                  const R fu = a == 0 ? g.fy : (a == 1 ? g.fz : g.fx);
                  const R fv = a == 0 ? g.fz : (a == 1 ? g.fx : g.fy);
                  const uint32_t mask = (1u << sh) - 1u;
                  const R scale = Num<R>::pow2m(g.lev) * (R)(1 << J.ptab_ssh) / (R)(1 << J.ptab_bsh);
                  const int S = 1 << J.ptab_ssh;
                  int iu = (int)Num<R>::floor_(((R)(cu & mask) + fu) * scale);
                  int iv = (int)Num<R>::floor_(((R)(cv & mask) + fv) * scale);
                  iu = iu < 0 ? 0 : (iu >= S ? S - 1 : iu);
                  iv = iv < 0 ? 0 : (iv >= S ? S - 1 : iv);
                  const ObsDev& O = J.obs[obs_o];
                  const uint32_t b0x = tab_blk & 1023u, b0y = (tab_blk >> 10) & 1023u, b0z = tab_blk >> 20;
                  const long long blk = (long long)b0x + (long long)J.ptab_nbx * ((long long)b0y + (long long)J.ptab_nby * b0z);
                  const long long i = O.tab_off + ((blk * O.tab_naxes + O.tab_slot[a]) * S + iv) * (long long)S + iu;
                  taup += ktab * (R)__ldg(J.ptab + i);
                  ev = taup > tau_cut ? EV_CUT : EV_ESCAPE;
                }
              }
            }
          }
        }
      } while (keep_stepping(ev, RT_PEEL_EV_BATCH));
    };
    const int key = st == P_LIVE ? akey : -1;
    const int k0 = __shfl_sync(FULL, key, __ffs(__ballot_sync(FULL, st == P_LIVE)) - 1);
    const bool same = __all_sync(FULL, st != P_LIVE || key == k0);
    if (RT_PEEL_AXIS && !TAB && same && k0 >= 0) {
      using A0 = std::integral_constant<int, 0>;
      using A1 = std::integral_constant<int, 1>;
      using A2 = std::integral_constant<int, 2>;
      if (k0 == 0) march(A0{}, std::false_type{});
      else if (k0 == 1) march(A0{}, std::true_type{});
      else if (k0 == 2) march(A1{}, std::false_type{});
      else if (k0 == 3) march(A1{}, std::true_type{});
      else if (k0 == 4) march(A2{}, std::false_type{});
      else march(A2{}, std::true_type{});
    } else {
      march(std::integral_constant<int, -1>{}, std::false_type{});
    }

    if (ev == EV_ESCAPE) {
      // the record's weighted phase function and pixel, as at the setup
      Geo<R> rg;
      R sdx, sdy, sdz, W;
      uint32_t meta;
      PeelIO<R>::get(Q.rec, (long long)rec_i, rg, sdx, sdy, sdz, W, meta);
      rg.lev = (int)(meta & 31u);
      const int bin = (int)((meta >> 5) & 255u);
      const JobDev& J = jobs[job];
      R pw = R(0);
      long long pix = 0;
      peel_setup<R>(J, obs_o, rg, sdx, sdy, sdz, W, Num<R>::gg(J.bins[bin]), bin, pw, pix);
      const R c = pw * Num<R>::exp_(-taup);
      if (c > R(0)) atomicAdd(J.images + pix, widen(c));
      book_d(SL, jobs, job, wid, L_PEEL, c);
    }
    if (ev == EV_ESCAPE || ev == EV_CUT) {
      book_u(SL, jobs, job, wid, U_PCROSS, npeel);
      st = P_DEAD;
    }
  }
  ledger_flush<R>(SL, jobs, wid, lane);
}

// ------------------------------------------------------------------------
// deterministic walk (diagnostic): the tracer's own node visits and face
// crossings, no physics
// ------------------------------------------------------------------------
template <typename R>
__global__ void walk_kernel(const JobDev* __restrict__ job, long long n_rays, const double* __restrict__ origins,
                            const double* __restrict__ dirs, long long max_seg, long long* __restrict__ cells,
                            double* __restrict__ lengths, long long* __restrict__ counts) {
  const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n_rays) return;
  const JobDev& J = *job;
  GridRegs G;
  G.node = J.node;
  G.rho64 = J.rho64;
  G.rx = J.root[0];
  G.ry = J.root[1];
  G.rz = J.root[2];
  const R dx = (R)dirs[3 * r], dy = (R)dirs[3 * r + 1], dz = (R)dirs[3 * r + 2];
  Geo<R> g;
  Cursor cur;
  g.rho = R(0);
  g.idx = 0u;
  if (!place_root(G, g, cur, (R)(origins[3 * r] / J.h0), (R)(origins[3 * r + 1] / J.h0),
                  (R)(origins[3 * r + 2] / J.h0), dx, dy, dz)) {
    counts[r] = -1;
    return;
  }
  const R ix = inv_abs(dx), iy = inv_abs(dy), iz = inv_abs(dz);
  // the tracers' stored path above the leaf, here in local memory
  uint32_t path[RT_ANC_MAX];
  AncPath P;
  P.a = path;
  P.stride = 1;
  P.cap = RT_ANC_MAX;
  P.n = RT_ANC_MAX;  // placed at the root: the descent stores the path
  uint32_t moved;
  long long k = 0;
  for (long long guard = 0; guard < 64ll * (1ll << 22); ++guard) {
    const uint32_t w = __ldg(G.node + cur.pending);
    const double r64 = Num<R>::load_rho64(G.rho64, cur.pending);
    if (w & RT_INTERIOR) {
      descend_step(g, cur, w, dx, dy, dz, P);
      continue;
    }
    settle_leaf(g, cur, w, r64);
    const Exit<R> E = exit_face(g, dx, dy, dz, ix, iy, iz);
    const R t = E.t;
    if (!Num<R>::finite(t)) break;
    if (t > R(0)) {
      if (k < max_seg) {
        cells[r * max_seg + k] = g.idx;
        lengths[r * max_seg + k] = (double)t * (double)Num<R>::pow2m(g.lev) * J.h0;
      }
      ++k;
    }
    if (!cross_face(G, g, cur, g.idx, E, t, true, dx, dy, dz, moved, P)) break;
  }
  counts[r] = k;
}

__global__ void philox_kernel(long long n, const uint32_t* __restrict__ ctr, const uint32_t* __restrict__ key,
                              uint32_t* __restrict__ out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
  const uint4 o = philox4x32_10(c, key[2 * i], key[2 * i + 1]);
  out[4 * i] = o.x;
  out[4 * i + 1] = o.y;
  out[4 * i + 2] = o.z;
  out[4 * i + 3] = o.w;
}

// ------------------------------------------------------------------------
// host launchers
// ------------------------------------------------------------------------
// dynamic shared memory of the stored paths (anc levels x the kernel's
// maximum block size, its path stride); the tracers' static shared memory
// plus this may exceed the default 48 KB, so the kernel is allowed that much
template <typename K>
static cudaError_t path_smem(K kernel, int max_block, int anc, size_t* bytes) {
  *bytes = (size_t)anc * (size_t)max_block * sizeof(uint32_t);
  if (*bytes == 0) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*bytes);
}

// the tracer for lanes that store anc levels of the path: the form that
// descends to the leaf exists for the untiled tracers of the continuous
// estimator, in FP64 in place of the level-by-level one
template <typename R, bool PEEL, int EST, bool HITS, int MODE, bool LEVELS, bool SPLIT>
static auto pick_tracer(int anc) {
  constexpr bool leaf_ok = MODE == 0 && EST == RT_EST_CONTINUOUS && !SPLIT;
  constexpr int deep = leaf_ok && sizeof(R) == 8 ? PATH_LEAF : PATH_LEVEL;
  const int form = path_form<R>(anc);
  return form == PATH_NONE   ? trace_kernel<R, PEEL, EST, HITS, MODE, LEVELS, SPLIT, PATH_NONE>
         : form == PATH_LEAF ? trace_kernel<R, PEEL, EST, HITS, MODE, LEVELS, SPLIT, leaf_ok ? PATH_LEAF : PATH_LEVEL>
                             : trace_kernel<R, PEEL, EST, HITS, MODE, LEVELS, SPLIT, deep>;
}

template <typename R, bool PEEL, int EST, bool HITS, int MODE, bool LEVELS, bool SPLIT>
static cudaError_t launch_mode(const JobDev* jobs, const ItemDev* items, int n_items, unsigned long long* counter,
                               long long total, const LaunchCfg& cfg, const PeelQueue& q, cudaStream_t s,
                               const TileRun& T) {
  auto k = pick_tracer<R, PEEL, EST, HITS, MODE, LEVELS, SPLIT>(cfg.anc);
  const int block = std::min(cfg.block, MaxThreads<R, MODE>::value);
  size_t dyn = 0;
  cudaError_t e = path_smem(k, MaxThreads<R, MODE>::value, cfg.anc, &dyn);
  if (e != cudaSuccess) return e;
  k<<<MODE == 2 ? cfg.blocks_tiled : cfg.blocks, block, dyn, s>>>(jobs, items, n_items, counter, total, cfg.refill,
                                                                  MODE == 2 ? 16 : cfg.ev_batch, q, T, cfg.anc);
  return cudaGetLastError();
}

template <typename R, bool PEEL, int EST, bool HITS, bool LEVELS = false>
static cudaError_t launch_t(const JobDev* jobs, const ItemDev* items, int n_items, unsigned long long* counter,
                            long long total, const LaunchCfg& cfg, const PeelQueue& q, cudaStream_t s, int mode,
                            const TileRun* tr) {
  TileRun T;
  memset(&T, 0, sizeof T);
  if (tr) T = *tr;
  if (mode == 1) return launch_mode<R, PEEL, EST, HITS, 1, LEVELS, false>(jobs, items, n_items, counter, total, cfg, q, s, T);
  if (mode == 2) return launch_mode<R, PEEL, EST, HITS, 2, LEVELS, false>(jobs, items, n_items, counter, total, cfg, q, s, T);
  return launch_mode<R, PEEL, EST, HITS, 0, LEVELS, false>(jobs, items, n_items, counter, total, cfg, q, s, T);
}

// resampling tracers: tiled modes only, continuous estimator, no hit counts
template <typename R, bool PEEL>
static cudaError_t launch_split(const JobDev* jobs, const ItemDev* items, int n_items, unsigned long long* counter,
                                long long total, const LaunchCfg& cfg, const PeelQueue& q, cudaStream_t s, int mode,
                                const TileRun* tr) {
  if (mode == 1)
    return launch_mode<R, PEEL, RT_EST_CONTINUOUS, false, 1, false, true>(jobs, items, n_items, counter, total, cfg,
                                                                          q, s, *tr);
  return launch_mode<R, PEEL, RT_EST_CONTINUOUS, false, 2, false, true>(jobs, items, n_items, counter, total, cfg, q,
                                                                        s, *tr);
}

template <typename R, int EST>
static cudaError_t launch_pe(bool peel, const JobDev* jobs, const ItemDev* items, int n_items,
                             unsigned long long* counter, long long total, const LaunchCfg& cfg,
                             const PeelQueue& q, cudaStream_t s, int mode, const TileRun* tr) {
  return peel ? launch_t<R, true, EST, false>(jobs, items, n_items, counter, total, cfg, q, s, mode, tr)
              : launch_t<R, false, EST, false>(jobs, items, n_items, counter, total, cfg, q, s, mode, tr);
}

// hit counting exists for the continuous estimator without peel-off (the
// Lambda iteration's noise mask)
cudaError_t launch_trace(int precision, bool peel, int estimator, bool hits, const JobDev* jobs_dev,
                         const ItemDev* items_dev, int n_items, unsigned long long* counter_dev, long long total,
                         const LaunchCfg& cfg, const PeelQueue& q, cudaStream_t s, int mode, const TileRun* tr,
                         bool levels, bool split) {
  const bool an = estimator == RT_EST_ANALOG;
  if ((mode == 1 || mode == 2) && !tr) return cudaErrorInvalidValue;
  if (split) {
    if (levels || hits || an || (mode != 1 && mode != 2)) return cudaErrorInvalidValue;
    if (precision == 64)
      return peel ? launch_split<double, true>(jobs_dev, items_dev, n_items, counter_dev, total, cfg, q, s, mode, tr)
                  : launch_split<double, false>(jobs_dev, items_dev, n_items, counter_dev, total, cfg, q, s, mode, tr);
    return peel ? launch_split<float, true>(jobs_dev, items_dev, n_items, counter_dev, total, cfg, q, s, mode, tr)
                : launch_split<float, false>(jobs_dev, items_dev, n_items, counter_dev, total, cfg, q, s, mode, tr);
  }
  if (levels) {
    // subiterations: dust traces with the continuous estimator, no peel-off
    if (peel || an) return cudaErrorInvalidValue;
    if (precision == 64)
      return hits ? launch_t<double, false, RT_EST_CONTINUOUS, true, true>(jobs_dev, items_dev, n_items, counter_dev,
                                                                           total, cfg, q, s, mode, tr)
                  : launch_t<double, false, RT_EST_CONTINUOUS, false, true>(jobs_dev, items_dev, n_items, counter_dev,
                                                                            total, cfg, q, s, mode, tr);
    return hits ? launch_t<float, false, RT_EST_CONTINUOUS, true, true>(jobs_dev, items_dev, n_items, counter_dev,
                                                                        total, cfg, q, s, mode, tr)
                : launch_t<float, false, RT_EST_CONTINUOUS, false, true>(jobs_dev, items_dev, n_items, counter_dev,
                                                                         total, cfg, q, s, mode, tr);
  }
  if (hits) {
    if (peel || an) return cudaErrorInvalidValue;
    return precision == 64
               ? launch_t<double, false, RT_EST_CONTINUOUS, true>(jobs_dev, items_dev, n_items, counter_dev, total, cfg,
                                                                  q, s, mode, tr)
               : launch_t<float, false, RT_EST_CONTINUOUS, true>(jobs_dev, items_dev, n_items, counter_dev, total, cfg,
                                                                 q, s, mode, tr);
  }
  if (precision == 64)
    return an ? launch_pe<double, RT_EST_ANALOG>(peel, jobs_dev, items_dev, n_items, counter_dev, total, cfg, q, s,
                                                 mode, tr)
              : launch_pe<double, RT_EST_CONTINUOUS>(peel, jobs_dev, items_dev, n_items, counter_dev, total, cfg, q,
                                                     s, mode, tr);
  return an ? launch_pe<float, RT_EST_ANALOG>(peel, jobs_dev, items_dev, n_items, counter_dev, total, cfg, q, s, mode,
                                              tr)
            : launch_pe<float, RT_EST_CONTINUOUS>(peel, jobs_dev, items_dev, n_items, counter_dev, total, cfg, q, s,
                                                  mode, tr);
}

size_t tile_record_bytes(int precision, bool wide) {
  return precision == 64 ? sizeof(TRec64) : (wide ? sizeof(TRec32W) : sizeof(TRec32));
}

// ------------------------------------------------------------------------
// counting sort of tile records by key
// ------------------------------------------------------------------------
__global__ void tile_hist_kernel(const uint32_t* __restrict__ key, long long n, int n_keys,
                                 unsigned long long* __restrict__ hist) {
  extern __shared__ unsigned int sh[];
  const bool use_sh = n_keys <= 8192;
  if (use_sh)
    for (int k = threadIdx.x; k < n_keys; k += blockDim.x) sh[k] = 0u;
  __syncthreads();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const uint32_t k = key[i];
    if (use_sh) atomicAdd(&sh[k], 1u);
    else atomicAdd(&hist[k], 1ull);
  }
  __syncthreads();
  if (use_sh)
    for (int k = threadIdx.x; k < n_keys; k += blockDim.x)
      if (sh[k]) atomicAdd(&hist[k], (unsigned long long)sh[k]);
}

// Exclusive prefix sums of hist within chunks of SCAN_KEYS, and the chunks'
// totals; the scatter adds the totals before its key's chunk.  (One block
// over all 262,144 keys of a peel-off queue took 118 to 400 us.)
static constexpr int SCAN_KEYS = 4096;
__global__ void __launch_bounds__(1024) tile_scan_kernel(unsigned long long* __restrict__ hist, int n,
                                                         unsigned long long* __restrict__ totals) {
  __shared__ unsigned long long part[32];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int b = blockIdx.x * SCAN_KEYS + 4 * t;
  unsigned long long v[4], sum = 0ull;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[i] = b + i < n ? hist[b + i] : 0ull;
    sum += v[i];
  }
  unsigned long long inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long x = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += x;
  }
  if (lane == 31) part[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    unsigned long long p = part[lane], q = p;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long x = __shfl_up_sync(0xFFFFFFFFu, q, o);
      if (lane >= o) q += x;
    }
    part[lane] = q - p;
    if (lane == 31) totals[blockIdx.x] = q;
  }
  __syncthreads();
  unsigned long long run = part[wid] + inc - sum;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (b + i < n) hist[b + i] = run;
    run += v[i];
  }
}

// scatter records to their key's range; lanes of a warp with equal keys
// take consecutive places with one atomic
__global__ void tile_scatter_kernel(const uint4* __restrict__ in, const uint32_t* __restrict__ key, long long n,
                                    const unsigned long long* __restrict__ count, int rec_u4, int n_chunks,
                                    const unsigned long long* __restrict__ totals, unsigned long long* __restrict__ offs,
                                    uint4* __restrict__ out) {
  extern __shared__ unsigned long long before[];  // records in the chunks of keys before each
  if (count) n = min(n, (long long)*count);
  for (int i = threadIdx.x; i < n_chunks; i += blockDim.x) before[i] = totals[i];
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long run = 0ull;
    for (int i = 0; i < n_chunks; ++i) {
      const unsigned long long v = before[i];
      before[i] = run;
      run += v;
    }
  }
  __syncthreads();
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long n_up = (n + 31) / 32 * 32;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n_up; i += stride) {
    const bool have = i < n;
    const uint32_t k = have ? key[i] : 0xFFFFFFFFu;
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, k);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(peers) - 1;
    unsigned long long base = 0ull;
    if (have && lane == leader) base = atomicAdd(&offs[k], (unsigned long long)__popc(peers));
    base = __shfl_sync(peers, base, leader);
    if (have) {
      const unsigned long long pos = before[k / SCAN_KEYS] + base + __popc(peers & ((1u << lane) - 1u));
      const uint4* src = in + i * rec_u4;
      uint4* dst = out + pos * rec_u4;
      for (int w = 0; w < rec_u4; ++w) dst[w] = src[w];
    }
  }
}

size_t tile_hist_bytes(int n_keys) {
  return sizeof(unsigned long long) * ((size_t)n_keys + (size_t)(n_keys + SCAN_KEYS - 1) / SCAN_KEYS + 1);
}

// the scan and scatter of a counting sort whose histogram is in hist
static cudaError_t sort_by_hist(const void* in, const uint32_t* key, long long n, const unsigned long long* count,
                                int rec_bytes, int n_keys, unsigned long long* hist, void* out, int grid,
                                cudaStream_t s) {
  const int nc = (n_keys + SCAN_KEYS - 1) / SCAN_KEYS;
  unsigned long long* totals = hist + n_keys;
  tile_scan_kernel<<<nc, 1024, 0, s>>>(hist, n_keys, totals);
  tile_scatter_kernel<<<grid, 512, sizeof(unsigned long long) * (size_t)nc, s>>>(
      static_cast<const uint4*>(in), key, n, count, rec_bytes / 16, nc, totals, hist, static_cast<uint4*>(out));
  return cudaGetLastError();
}

cudaError_t tile_sort(const void* in, const uint32_t* key, long long n, int rec_bytes, int n_keys,
                      unsigned long long* hist_dev, void* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (rec_bytes % 16) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(hist_dev, 0, sizeof(unsigned long long) * (size_t)n_keys, s);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int B = 512;
  const long long want = (n + B - 1) / B;
  const int G = (int)std::min<long long>(want, (long long)sms * 4);
  const size_t shb = n_keys <= 8192 ? sizeof(unsigned int) * (size_t)n_keys : 0;
  tile_hist_kernel<<<G, B, shb, s>>>(key, n, n_keys, hist_dev);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return sort_by_hist(in, key, n, nullptr, rec_bytes, n_keys, hist_dev, out, G, s);
}

bool descents_counted() { return RT_COUNT_DESCENTS != 0; }

cudaError_t descent_counts(unsigned long long out[2], bool reset) {
  cudaError_t e = cudaMemcpyFromSymbol(out, g_descents, 2 * sizeof(unsigned long long));
  if (e == cudaSuccess && reset) {
    const unsigned long long z[2] = {0ull, 0ull};
    e = cudaMemcpyToSymbol(g_descents, z, sizeof z);
  }
  return e;
}

size_t peel_record_bytes(int precision) { return precision == 64 ? sizeof(PeelRec64) : sizeof(PeelRec32); }

// sort key of a deferred peel-off record: the block of 2^bs root cells
// holding the scattering point, x fastest, clamped to the nbx x nby x nbz
// blocks of the first job's root grid; and the keys' histogram
template <typename R>
__global__ void __launch_bounds__(512) peel_key_kernel(const void* __restrict__ rec, long long n,
                                                       const unsigned long long* __restrict__ count, int bs, int nbx,
                                                       int nby, int nbz, uint32_t* __restrict__ key, int n_keys,
                                                       unsigned long long* __restrict__ hist) {
  extern __shared__ unsigned int sh[];
  const bool use_sh = n_keys <= 8192;
  if (use_sh)
    for (int k = threadIdx.x; k < n_keys; k += blockDim.x) sh[k] = 0u;
  __syncthreads();
  if (count) n = min(n, (long long)*count);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    uint4 a;
    uint32_t meta;
    if (sizeof(R) == 4) {
      const uint4* p = reinterpret_cast<const uint4*>(static_cast<const PeelRec32*>(rec) + i);
      a = __ldg(p);
      meta = __ldg(&p[2].w);
    } else {
      const PeelRec64* r = static_cast<const PeelRec64*>(rec) + i;
      a = __ldg(reinterpret_cast<const uint4*>(&r->cx));
      meta = __ldg(&r->meta);
    }
    const int shf = (int)(meta & 31u) + bs;
    const uint32_t bx = min(a.x >> shf, (uint32_t)(nbx - 1));
    const uint32_t by = min(a.y >> shf, (uint32_t)(nby - 1));
    const uint32_t bz = min(a.z >> shf, (uint32_t)(nbz - 1));
    const uint32_t k = bx + (uint32_t)nbx * (by + (uint32_t)nby * bz);
    key[i] = k;
    if (use_sh) atomicAdd(&sh[k], 1u);
    else atomicAdd(&hist[k], 1ull);
  }
  __syncthreads();
  if (use_sh)
    for (int k = threadIdx.x; k < n_keys; k += blockDim.x)
      if (sh[k]) atomicAdd(&hist[k], (unsigned long long)sh[k]);
}

cudaError_t peel_sort(int precision, const void* rec, long long n, const unsigned long long* count, int bs, int nbx,
                      int nby, int nbz, uint32_t* key, unsigned long long* hist, void* out, int sm_count,
                      cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int n_keys = nbx * nby * nbz;
  cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * (size_t)n_keys, s);
  if (e != cudaSuccess) return e;
  const int B = 512;
  // a count on the device may be far below n: no more blocks than fill the GPU
  const int G = (int)std::min<long long>((n + B - 1) / B, (long long)sm_count * 4);
  const size_t shb = n_keys <= 8192 ? sizeof(unsigned int) * (size_t)n_keys : 0;
  if (precision == 64) peel_key_kernel<double><<<G, B, shb, s>>>(rec, n, count, bs, nbx, nby, nbz, key, n_keys, hist);
  else peel_key_kernel<float><<<G, B, shb, s>>>(rec, n, count, bs, nbx, nby, nbz, key, n_keys, hist);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return sort_by_hist(rec, key, n, count, (int)peel_record_bytes(precision), n_keys, hist, out, G, s);
}

template <typename R, bool TAB>
static cudaError_t launch_peel_t(const JobDev* jobs, const PeelQueue& q, unsigned long long* work, int n_obs_max,
                                 int refill, cudaStream_t s, int anc) {
  int dev = 0, sms = 0, occ = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int form = path_form<R>(anc);
  auto k = form == PATH_NONE   ? peel_kernel<R, TAB, PATH_NONE>
           : form == PATH_LEAF ? peel_kernel<R, TAB, PATH_LEAF>
                               : peel_kernel<R, TAB, sizeof(R) == 8 ? PATH_LEAF : PATH_LEVEL>;
  size_t dyn = 0;
  cudaError_t e = path_smem(k, 256, anc, &dyn);
  if (e != cudaSuccess) return e;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, 256, dyn) != cudaSuccess || occ < 1) occ = 1;
  k<<<sms * occ, 256, dyn, s>>>(jobs, q, work, n_obs_max, refill, anc);
  return cudaGetLastError();
}

cudaError_t launch_peel(int precision, const JobDev* jobs_dev, const PeelQueue& q, unsigned long long* work_dev,
                        int n_obs_max, int refill, cudaStream_t s, int anc) {
  if (q.cap <= 0 || n_obs_max <= 0) return cudaSuccess;
  return precision == 64 ? launch_peel_t<double, false>(jobs_dev, q, work_dev, n_obs_max, refill, s, anc)
                         : launch_peel_t<float, false>(jobs_dev, q, work_dev, n_obs_max, refill, s, anc);
}

cudaError_t launch_peel_tab(int precision, const JobDev* jobs_dev, const PeelQueue& q, unsigned long long* work_dev,
                            int n_obs_max, int refill, cudaStream_t s, int anc) {
  if (q.cap <= 0 || n_obs_max <= 0) return cudaSuccess;
  return precision == 64 ? launch_peel_t<double, true>(jobs_dev, q, work_dev, n_obs_max, refill, s, anc)
                         : launch_peel_t<float, true>(jobs_dev, q, work_dev, n_obs_max, refill, s, anc);
}

// ------------------------------------------------------------------------
// accelerated peel-off tables (Sect. 2.4): one thread per entry marches in
// FP64 from the tile centre to the model border and sums density x length
// ------------------------------------------------------------------------
__global__ void peel_table_kernel(const JobDev* __restrict__ job, PeelTabSpec S, long long n,
                                  double* __restrict__ out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int o = 0;
  while (o + 1 < S.n_obs && S.off[o + 1] <= i) ++o;
  long long r = i - S.off[o];
  const int T = S.tiles;
  const int iu = (int)(r % T);
  r /= T;
  const int iv = (int)(r % T);
  r /= T;
  const int ai = (int)(r % S.n_axes[o]);
  const long long blk = r / S.n_axes[o];
  const int a = S.axes[o][ai], a1 = (a + 1) % 3, a2 = (a + 2) % 3;
  const JobDev& J = *job;
  const int Rr[3] = {(int)J.root[0], (int)J.root[1], (int)J.root[2]};
  const int b[3] = {(int)(blk % S.nb[0]), (int)((blk / S.nb[0]) % S.nb[1]), (int)(blk / ((long long)S.nb[0] * S.nb[1]))};
  const double* k = S.k[o];
  double c[3];
  c[a] = k[a] > 0 ? fmin((double)(b[a] + 1) * S.block, (double)Rr[a]) : (double)b[a] * S.block;
  const double w = (double)S.block / T;
  const double u0 = (double)b[a1] * S.block + iu * w, v0 = (double)b[a2] * S.block + iv * w;
  if (u0 >= Rr[a1] || v0 >= Rr[a2]) {
    out[i] = 0.0;
    return;
  }
  c[a1] = 0.5 * (u0 + fmin(u0 + w, (double)Rr[a1]));
  c[a2] = 0.5 * (v0 + fmin(v0 + w, (double)Rr[a2]));
  GridRegs G;
  G.node = J.node;
  G.rho64 = J.rho64;
  G.rx = J.root[0];
  G.ry = J.root[1];
  G.rz = J.root[2];
  Geo<double> g;
  Cursor cur;
  double col = 0.0;
  if (place_root(G, g, cur, c[0], c[1], c[2], k[0], k[1], k[2])) {
    const double ix = inv_abs(k[0]), iy = inv_abs(k[1]), iz = inv_abs(k[2]);
    for (int pass = 0; pass < (1 << 26); ++pass) {
      const uint32_t wd = G.node[cur.pending];
      const double r64 = G.rho64[cur.pending];
      if (wd & RT_INTERIOR) {
        descend_step(g, cur, wd, k[0], k[1], k[2]);
        continue;
      }
      settle_leaf(g, cur, wd, r64);
      const Exit<double> E = exit_face(g, k[0], k[1], k[2], ix, iy, iz);
      if (!Num<double>::finite(E.t)) break;
      col += Num<double>::down(g.rho, g.lev) * E.t;
      if (!cross_face(G, g, cur, g.idx, E, k[0], k[1], k[2])) break;
    }
  }
  out[i] = col;
}

cudaError_t build_peel_table(const JobDev* job_dev, const PeelTabSpec& spec, double* table, cudaStream_t s) {
  const long long n = spec.off[spec.n_obs];
  if (n <= 0) return cudaSuccess;
  const int B = 128;
  peel_table_kernel<<<(unsigned)((n + B - 1) / B), B, 0, s>>>(job_dev, spec, n, table);
  return cudaGetLastError();
}

// blocks per SM of the plain tracer (MODE 0 or 2) with the same path levels
template <typename R, bool PEEL, int MODE>
static cudaError_t occ_t(int block, int* n, int anc) {
  auto k = pick_tracer<R, PEEL, RT_EST_CONTINUOUS, false, MODE, false, false>(anc);
  size_t dyn = 0;
  cudaError_t e = path_smem(k, MaxThreads<R, MODE>::value, anc, &dyn);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k, std::min(block, MaxThreads<R, MODE>::value), dyn);
}

template <typename R, bool PEEL>
static cudaError_t occ_mode(int block, int* n, int mode, int anc) {
  return mode == 2 ? occ_t<R, PEEL, 2>(block, n, anc) : occ_t<R, PEEL, 0>(block, n, anc);
}

cudaError_t trace_occupancy(int precision, bool peel, int block, int* blocks_per_sm, int mode, int anc) {
  if (precision == 64)
    return peel ? occ_mode<double, true>(block, blocks_per_sm, mode, anc)
                : occ_mode<double, false>(block, blocks_per_sm, mode, anc);
  return peel ? occ_mode<float, true>(block, blocks_per_sm, mode, anc)
              : occ_mode<float, false>(block, blocks_per_sm, mode, anc);
}

cudaError_t launch_walk(int precision, const JobDev* job_dev, long long n_rays, const double* origins,
                        const double* dirs, long long max_seg, long long* cells, double* lengths, long long* counts,
                        cudaStream_t s) {
  const int B = 128;
  const unsigned G = (unsigned)((n_rays + B - 1) / B);
  if (G == 0) return cudaSuccess;
  if (precision == 64) walk_kernel<double><<<G, B, 0, s>>>(job_dev, n_rays, origins, dirs, max_seg, cells, lengths, counts);
  else walk_kernel<float><<<G, B, 0, s>>>(job_dev, n_rays, origins, dirs, max_seg, cells, lengths, counts);
  return cudaGetLastError();
}

// L2 read bandwidth (diagnostic for the rooflines): every thread streams
// 16-byte loads cached in L2 only (ld.global.cg) over a buffer that fits in
// L2, `reps` times; the XOR of the words is stored only if it equals a value
// a zeroed buffer cannot give, which keeps the loads
__global__ void l2_read_kernel(const uint4* __restrict__ p, long long n, int reps, unsigned* __restrict__ sink) {
  unsigned acc = 0u;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (int r = 0; r < reps; ++r)
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
      const uint4 v = __ldcg(p + i);
      acc ^= v.x ^ v.y ^ v.z ^ v.w;
    }
  if (acc == 0x9E3779B9u) sink[0] = acc;
}

cudaError_t launch_l2_read(const void* buf, long long bytes, int reps, int sm_count, cudaStream_t s) {
  const long long n = bytes / 16;
  if (n <= 0) return cudaSuccess;
  l2_read_kernel<<<sm_count * 8, 256, 0, s>>>(static_cast<const uint4*>(buf), n, reps,
                                              const_cast<unsigned*>(static_cast<const unsigned*>(buf)));
  return cudaGetLastError();
}

cudaError_t launch_philox(long long n, const uint32_t* ctr, const uint32_t* key, uint32_t* out, cudaStream_t s) {
  const int B = 256;
  const unsigned G = (unsigned)((n + B - 1) / B);
  if (G == 0) return cudaSuccess;
  philox_kernel<<<G, B, 0, s>>>(n, ctr, key, out);
  return cudaGetLastError();
}

}  // namespace rtk
