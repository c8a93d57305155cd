// trace.cu -- persistent ray-tracing kernel (Sec. 2.1-2.2, Steps 1-5 of
// Sec. 3.1) for one or many grids at once.
//
// Work model.  Every lane of the persistent grid carries at most one photon
// package.  A lane without a package takes a ticket from a global counter
// (one atomic per warp).  Tickets below n_roots are root packages (Step 1:
// source = ticket / N_pix, pixel = ticket % N_pix, P = 1 in units of the
// source's Ndot / N_pix) and need no memory; higher tickets name queue slots
// that split packages publish.  When a package splits (Step 3e) its lane
// keeps child 0 and hands children 1-3 to lanes of its warp whose package
// ended in the same round (no package, no ticket), by warp shuffles; the
// rest go to the queue (one atomic per warp reserves the slots), where each
// 32-byte record's tag word is stored last, after a fence, and
// polled with acquire loads.  An outstanding-package counter
// (+3 per split, -1 per finished package) tells idle warps when the trace is
// over.  Every wait is bounded: a warp that sees no change of the counter for
// timeout_ns sets RT_ERR_TIMEOUT and leaves; a package that takes more steps
// than a ray can cross planes sets RT_ERR_STATE.  Nothing traps.
//
// Per segment (Steps 3d-3i): next crossing r_next = min_i t_i (Eq. "trace"),
// split test r_next > R_split(l) (Eq. "split"), tau = sigma n_HI dr
// (Eq. "dtau"), dP = P (1 - e^-tau) (Eq. "flux"), k_ph += P w dr phi(tau)
// with phi = (1 - e^-tau)/tau (Eq. "kph"), Gamma += k_ph (E - 13.6 eV)
// (Eq. "gamma"), then termination at tau_tot > -ln f_term with the residual
// absorbed in place, and exit at the box boundary.
//
// Finite speed of light (Step 3j; the kernel instantiated with FSL): a
// package of age a (traces since its emission) halts where its crossing
// radius would pass rlim[a]; the cut segment is deposited, the termination
// test comes first, and the package is appended to an output store with its
// cell.  The next trace's tickets n_roots .. n_roots + n_res - 1 name the
// stored packages, which continue from their cells.  This instantiation
// queues every child 1-3, in 48-byte records that carry the age.
#include <type_traits>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "f2.cuh"
#include "healpix.cuh"
#include "rt_internal.cuh"

#ifndef TRACE_MIN_BLOCKS
#define TRACE_MIN_BLOCKS 2
#endif

namespace rtg {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kShInst = 64;  // grids whose level counters and fallback counts a block keeps in shared memory
static_assert(kBlkGrids <= kShInst, "a grid with a budget row has its counters in shared memory");
constexpr int kBlock = 256;  // threads per block of the trace kernel

// What ends a lane's part of a queue visit.  EV_RARE: the next segment needs
// the full decision; EV_TERM: the optical depth is at or near the termination
// (the FP32 walker leaves both to a stage after the visit's segments).
enum Event { EV_NONE = 0, EV_SPLIT, EV_DONE, EV_HALT, EV_RARE, EV_TERM };
enum Start { NO_START = 0, START_CHILD, START_ROOT, START_RESUMED };
constexpr int kAcc = 5;  // budget sums per grid: emitted, absorbed, escaped, resumed, halted

// Position of the set bit of rank n (0 = lowest) in m; m holds more than n
// set bits.  A binary search on the population counts of the low halves.
__device__ __forceinline__ int nth_set_bit(unsigned m, unsigned n) {
  int pos = 0;
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) {
    const unsigned low = m & ((1u << w) - 1u);
    const unsigned c = (unsigned)__popc(low);
    if (c <= n) {
      n -= c;
      m >>= w;
      pos += w;
    } else {
      m = low;
    }
  }
  return pos;
}

// Photon budget of one lane for the grid it is working on; lives in shared
// memory (one slot per thread) and is touched only at package events.
struct LaneAcc {
  double emitted, absorbed, escaped, resumed, halted;
  unsigned long long segments;
  unsigned int fallbacks, fallbacks_tau;
  int inst;
  // of the lane's package (FP32 walker), read only between queue visits and so
  // kept out of registers: P, optical depth and its error bound at the start,
  // the radius of the next full decision, segments so far, and the planes
  // that a segment left at EV_TERM crosses
  float Pstart, tau0, tau_err, lim;
  int steps, mask;
  float cover;  // covering factor of the last segment (where traced with one)
  double n[3];  // the direction in FP64, once a decision has needed it (level and pix it is of)
  uint32_t n_level, n_pix;
  // 120 bytes = 30 banks: the 8-byte accesses of a half-warp to one field
  // fall on 16 different bank pairs (a 64-byte stride puts them on two)
};
static_assert(sizeof(LaneAcc) == 120, "conflict-free stride of the per-lane sums");

// A block's budget sums per grid for the first kBlkGrids grids of the
// launch: its rows of TraceArgs.blk (global memory, kBlkRow words per grid)
// and, for the rare fallback counts, a table in shared memory.  A lane that
// moves to a package of another grid adds its sums to the rows with
// reductions whose results it does not wait for; the block adds its rows
// into the grids' sums once at the end.  (Shared-memory FP64 atomics, which
// return their result, cost the 64-grid batch 11 % of its trace time.)
struct BlockBudget {
  double* rows;             // [nrows][kBlkRow]: emitted, absorbed, escaped, resumed, halted, segments
  int nrows;                // min(grids of the launch, kBlkGrids)
  unsigned int* fb;         // [kShInst][2]: fallbacks, fallbacks_tau
};

// Grids beyond the block's rows (rare: batches of more than kBlkGrids
// grids) flush to the grid's sums directly, out of line.
__device__ __noinline__ void acc_flush_global(const LaneAcc& a, const TraceArgs& A) {
  const InstDev& I = A.inst[a.inst];
  if (a.emitted != 0.0) atomicAdd(&I.acc[0], a.emitted);
  if (a.absorbed != 0.0) atomicAdd(&I.acc[1], a.absorbed);
  if (a.escaped != 0.0) atomicAdd(&I.acc[2], a.escaped);
  if (a.resumed != 0.0) atomicAdd(&I.acc[3], a.resumed);
  if (a.halted != 0.0) atomicAdd(&I.acc[4], a.halted);
  if (a.segments) atomicAdd(&I.cnt[kCntSegments], a.segments);
  if (a.fallbacks) atomicAdd(&I.cnt[kCntFallbacks], (unsigned long long)a.fallbacks);
  if (a.fallbacks_tau) atomicAdd(&I.cnt[kCntFallbacksTau], (unsigned long long)a.fallbacks_tau);
}
__device__ __forceinline__ void acc_flush(LaneAcc& a, const TraceArgs& A, const BlockBudget& bb) {
  if (a.inst >= 0 && a.inst < bb.nrows) {
    // straight-line reductions (adding zeros costs less than branching)
    double* t = bb.rows + kBlkRow * a.inst;
    red_add(&t[0], a.emitted);
    red_add(&t[1], a.absorbed);
    red_add(&t[2], a.escaped);
    if (a.resumed != 0.0 || a.halted != 0.0) {
      red_add(&t[3], a.resumed);
      red_add(&t[4], a.halted);
    }
    red_add(reinterpret_cast<unsigned long long*>(&t[kAcc]), a.segments);
    if (a.fallbacks | a.fallbacks_tau) {
      atomicAdd(&bb.fb[2 * a.inst], a.fallbacks);
      atomicAdd(&bb.fb[2 * a.inst + 1], a.fallbacks_tau);
    }
  } else if (a.inst >= 0) {
    acc_flush_global(a, A);
  }
  a.emitted = a.absorbed = a.escaped = a.resumed = a.halted = 0.0;
  a.segments = 0;
  a.fallbacks = 0;
  a.fallbacks_tau = 0;
}

// Switch the lane's budget to grid `inst`, flushing the previous grid's sums
// (with the segments counted since the last switch).
__device__ __forceinline__ void acc_switch(LaneAcc& a, unsigned& nseg, int inst, const TraceArgs& A,
                                           const BlockBudget& bb) {
  if (a.inst != inst) {
    a.segments += nseg;
    nseg = 0;
    acc_flush(a, A, bb);
    a.inst = inst;
  }
}

// A warp's state while it has nothing to trace: the outstanding count last
// seen, when it was first seen, and how long to sleep (ns; doubles up to 1 us).
struct IdleWarp {
  long long seen_out;
  uint64_t seen_ns;
  unsigned backoff;
};

struct LevelCounters {
  unsigned int* cnt;        // [kShInst][kLevels]
  unsigned long long* hsh;  // [kShInst][kLevels]
  // Count n packages (level, pix0 .. pix0 + n - 1) of a source; the
  // checksum terms only when requested.
  __device__ __forceinline__ void add(const TraceArgs& A, int inst, int local, int level, uint32_t pix0,
                                      uint32_t n) {
    unsigned long long h = 0;
    if (A.checksums)
      for (uint32_t k = 0; k < n; ++k) h += pkg_hash((uint32_t)local, (uint32_t)level, pix0 + k);
    if (inst < kShInst) {
      atomicAdd(&cnt[inst * kLevels + level], n);
      if (A.checksums) atomicAdd(&hsh[inst * kLevels + level], h);
    } else {
      atomicAdd(&A.inst[inst].cnt[level], (unsigned long long)n);
      if (A.checksums) atomicAdd(&A.inst[inst].cnt[kLevels + level], h);
    }
  }
};

// ---------------------------------------------------------------------------
// FP64 walker: every decision (cell of a point, next crossing, split,
// termination) is evaluated with explicitly rounded FP64 operations in the
// order a plain FP64 evaluation of the method's formulas uses.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int cell_of64(double u, double n) {
  if (n > 0) return (int)floor(u);
  if (n < 0) return (int)ceil(u) - 1;
  return (int)floor(u);
}
__device__ __forceinline__ double next_t64(int c, double s, double n) {
  if (n > 0) return __ddiv_rn(__dsub_rn((double)(c + 1), s), n);
  if (n < 0) return __ddiv_rn(__dsub_rn((double)c, s), n);
  return __longlong_as_double(0x7ff0000000000000LL);  // +inf
}

// The FP64 pipe (1/64 of the FP32 rate) bounds this walker: distances are
// compared as integers (positive doubles order like their bit patterns), the
// planes of an axis are counted in FP64, and the next cell's density is loaded
// before the absorption.  Trace of the 128^3 Stroemgren snapshot 4.1 -> 3.2 ms.
struct Walk64 {
  using Rec = Rec64;
  template <bool FSL> using Q = Rec64;  // queue record
  uint32_t src, level, pix;
  uint32_t age;   // traces since emission (finite speed of light)
  double r, P, tau, Pstart;
  double rlim;    // halting radius of this age
  double rsp;     // split radius (+inf: the package does not split)
  double s0, s1, s2, n0, n1, n2, t0, t1, t2;
  double b0, b1, b2;  // the next plane of each axis
  double nh;          // absorber density of the current cell
  int c0, c1, c2;
  int nx, ny, nz, steps;
  int idx;
  unsigned nseg;
  const double* nhi;
  double* K;
  double* G;
  double sdx, w, rw, heat;

  __device__ __forceinline__ bool inside() const {
    return c0 >= 0 && c0 < nx && c1 >= 0 && c1 < ny && c2 >= 0 && c2 < nz;
  }
  __device__ __forceinline__ int inst(const TraceArgs& A) const { return A.src[src].inst; }
  __device__ __forceinline__ double unit(const TraceArgs& A) const { return A.src[src].unit; }
  __device__ __forceinline__ int lvl() const { return (int)level; }
  // P of a new package of source S (finite speed of light)
  __device__ __forceinline__ double emit(const SourceDev& S) {
    P = S.p0;
    return P;
  }

  __device__ __forceinline__ void bind(const TraceArgs& A) {
    const SourceDev& S = A.src[src];
    s0 = S.s[0]; s1 = S.s[1]; s2 = S.s[2];
    sdx = S.sdx; w = S.w; rw = S.rw; heat = S.heat;
    const InstDev& I = A.inst[S.inst];
    nx = I.nx; ny = I.ny; nz = I.nz;
    // the absorber and accumulators of the package's photon type (Sec. 3.2)
    const int t = S.type;
    nhi = (const double*)(t == 0 ? I.nhi : I.nhe[t - 1]);
    K = (double*)(t == 0 ? I.K : I.Khe[t - 1]);
    G = (double*)(t == 0 ? I.G : I.Ghe[t - 1]);
    double n[3];
    pix2vec64((int)level, pix, n);
    n0 = n[0]; n1 = n[1]; n2 = n[2];
    Pstart = P;
    steps = 0;
  }
  // the plane that cell c's ray meets next on an axis, and its distance
  __device__ __forceinline__ static void axis(int c, double s, double n, double& b, double& t) {
    b = (double)(n > 0 ? c + 1 : c);
    t = n != 0 ? __ddiv_rn(__dsub_rn(b, s), n) : __longlong_as_double(0x7ff0000000000000LL);
  }
  // Steps 3a-3b: direction and cell at radius r, false outside the box.  A
  // package continued from the previous trace (given) is in the cell it
  // halted in.
  template <bool FSL>
  __device__ __forceinline__ bool start(const TraceArgs& A, LaneAcc&, bool given, uint32_t cell) {
    bind(A);
    if (FSL && given) {
      c0 = (int)(cell % (uint32_t)nx);
      c1 = (int)((cell / (uint32_t)nx) % (uint32_t)ny);
      c2 = (int)(cell / ((uint32_t)nx * (uint32_t)ny));
    } else {
      c0 = cell_of64(__dadd_rn(s0, __dmul_rn(r, n0)), n0);
      c1 = cell_of64(__dadd_rn(s1, __dmul_rn(r, n1)), n1);
      c2 = cell_of64(__dadd_rn(s2, __dmul_rn(r, n2)), n2);
      if (!inside()) return false;
    }
    idx = c0 + nx * (c1 + ny * c2);
    nh = __ldg(&nhi[idx]);
    axis(c0, s0, n0, b0, t0);
    axis(c1, s1, n1, b1, t1);
    axis(c2, s2, n2, b2, t2);
    rsp = (int)level < A.max_level ? A.rsplit[level] : __longlong_as_double(0x7ff0000000000000LL);
    return true;
  }
  __device__ __forceinline__ void set_rlim(const TraceArgs& A) {
    if ((int)age < A.n_ages) rlim = A.rlim64[age];
    else { set_status(A.ctl, RT_ERR_STATE); rlim = 0.0; }
  }

  __device__ __forceinline__ void load(const Rec& q) {
    r = q.r; P = q.P; tau = q.tau; src = q.src; pix = q.pix; level = q.level & 15u; age = q.level >> 4;
  }
  // Record of child cpix (level + 1, P/4, same radius, optical depth and age).
  __device__ __forceinline__ Rec make_child(uint32_t cpix) const {
    Rec c;
    c.r = r; c.P = P * 0.25; c.tau = tau; c.src = src; c.pix = cpix; c.level = (level + 1) | (age << 4); c.tag = 0;
    return c;
  }
  __device__ __forceinline__ static uint32_t cell_of_record(const Rec& q) { return q.tag; }
  // A halted package as the next trace continues it (one trace older).
  __device__ __forceinline__ void store_halted(Rec* q) const {
    Rec c;
    c.r = r; c.P = P; c.tau = tau; c.src = src; c.pix = pix; c.level = level | ((age + 1) << 4);
    c.tag = (uint32_t)(c0 + nx * (c1 + ny * c2));
    *q = c;
  }
  // A record's payload into its queue slot; the tag that completes it follows
  // a fence.  (The age travels in the level word either way.)
  template <bool FSL>
  __device__ __forceinline__ static void put(Rec* q, const Rec& c) {
    __stcg(reinterpret_cast<double2*>(&q->r), make_double2(c.r, c.P));
    __stcg(reinterpret_cast<double*>(&q->tau), c.tau);
    __stcg(reinterpret_cast<uint2*>(&q->src), make_uint2(c.src, c.pix));
    __stcg(&q->level, c.level);
  }
  template <bool FSL>
  __device__ __forceinline__ static uint32_t tag_of(const Rec&, uint32_t epoch) { return epoch; }
  // Poll with an acquire load of the tag: the payload reads that follow a
  // successful poll are ordered after it without a fence.
  template <bool FSL>
  __device__ __forceinline__ static bool poll(const Rec* q, uint32_t epoch, Rec& o) {
    if (ld_acquire_u32(&q->tag) != epoch) return false;
    const double2 a = __ldcg(reinterpret_cast<const double2*>(&q->r));    // r, P
    const double2 b = __ldcg(reinterpret_cast<const double2*>(&q->tau));  // tau, (src, pix)
    const uint2 c = __ldcg(reinterpret_cast<const uint2*>(&q->level));    // level, tag
    const unsigned long long sp = (unsigned long long)__double_as_longlong(b.y);
    o.r = a.x; o.P = a.y; o.tau = b.x;
    o.src = (uint32_t)(sp & 0xffffffffu);
    o.pix = (uint32_t)(sp >> 32);
    o.level = c.x;
    return true;
  }
  // Every lane takes the record that lane `from` holds (all lanes call it).
  __device__ __forceinline__ static void shfl_rec(Rec& c, int from) {
    c.r = __shfl_sync(0xffffffffu, c.r, from);
    c.P = __shfl_sync(0xffffffffu, c.P, from);
    c.tau = __shfl_sync(0xffffffffu, c.tau, from);
    c.src = __shfl_sync(0xffffffffu, c.src, from);
    c.pix = __shfl_sync(0xffffffffu, c.pix, from);
    c.level = __shfl_sync(0xffffffffu, c.level, from);
  }
  __device__ __forceinline__ static Rec root_rec(uint32_t gsrc, uint32_t lvl0, uint32_t p) {
    Rec c;
    c.r = 0.0; c.P = 1.0; c.tau = 0.0; c.src = gsrc; c.pix = p; c.level = lvl0; c.tag = 0;
    return c;
  }
  __device__ __forceinline__ void become_child0() {
    level += 1; pix = 4u * pix; P = P * 0.25;
  }

  __device__ __forceinline__ static long long bits(double v) { return __double_as_longlong(v); }
  // past the axis' next plane
  __device__ __forceinline__ static void cross(double n, double s, double& b, double& t, int& c) {
    const bool up = bits(n) > 0;
    b = __dadd_rn(b, up ? 1.0 : -1.0);
    t = __ddiv_rn(__dsub_rn(b, s), n);
    c += up ? 1 : -1;
  }

  // One segment.  Returns EV_SPLIT before traversing a cell whose exit radius
  // exceeds R_split, EV_DONE when the package is absorbed or leaves the box,
  // EV_HALT (FSL) when it has travelled to its halting radius.
  template <bool FSL>
  __device__ __forceinline__ int step(const TraceArgs& A, LaneAcc& acc) {
    // distances are positive or +0 here
    long long u = bits(t0) < bits(t1) ? bits(t0) : bits(t1);
    if (bits(t2) < u) u = bits(t2);
    if (u > bits(rsp)) return EV_SPLIT;
    const double rn = __longlong_as_double(u);
    const bool m0 = bits(t0) == u, m1 = bits(t1) == u, m2 = bits(t2) == u;
    const bool halt = FSL && u > bits(rlim);  // Step 3j
    double dr = __dsub_rn(halt ? rlim : rn, r);
    if (bits(dr) < 0) dr = 0.0;
    const int at = idx;
    const double n_abs = nh, r0 = r;
    const int k0 = c0, k1 = c1, k2 = c2;
    bool out = false;
    if (!halt) {
      // cross first: the next cell's density arrives during the absorption
      if (m0) cross(n0, s0, b0, t0, c0);
      if (m1) cross(n1, s1, b1, t1, c1);
      if (m2) cross(n2, s2, b2, t2, c2);
      r = rn;
      out = !inside();
      if (!out) {
        idx = c0 + nx * (c1 + ny * c2);
        nh = __ldg(&nhi[idx]);
      }
    }
    const double dtau = __dmul_rn(__dmul_rn(sdx, n_abs), dr);
    const double am = -expm1(-dtau);
    const double phi = bits(dtau) > 0 ? am / dtau : 1.0;
    double kadd = P * w * dr * phi;
    // covering factor (Eq. "fc"): pixel width at r, midpoint to nearest face
    double fcv = 1.0;
    if (A.fc) {
      const double L = r0 * A.theta[level];
      if (L > 0.0) {
        const double rm = r0 + 0.5 * dr;
        const double d = fmax(fabs(s0 + n0 * rm - (k0 + 0.5)),
                              fmax(fabs(s1 + n1 * rm - (k1 + 0.5)), fabs(s2 + n2 * rm - (k2 + 0.5))));
        const double f = 0.5 + (0.5 - d) / L;
        fcv = fmin(1.0, f * f);
      }
      kadd *= fcv;
    }
    if (bits(dr) > 0) nseg++;
    P = fma(-P, am, P);
    tau = __dadd_rn(tau, dtau);
    const bool term = bits(tau) > bits(A.tau_term);
    if (term) kadd += P * rw / n_abs * fcv;  // the residual, absorbed here
    red_add(&K[at], kadd);
    if (bits(heat) != 0) red_add(&G[at], kadd * heat);
    if (term) {
      acc.absorbed += Pstart * unit(A);
      return EV_DONE;
    }
    if (halt) {
      r = rlim;
      const double u1 = unit(A);
      acc.absorbed += (Pstart - P) * u1;
      acc.halted += P * u1;
      return EV_HALT;
    }
    if (out) {
      const double u1 = unit(A);
      acc.absorbed += (Pstart - P) * u1;
      acc.escaped += P * u1;
      return EV_DONE;
    }
    if (++steps > A.max_steps) {
      set_status(A.ctl, RT_ERR_STATE);
      const double u1 = unit(A);
      acc.absorbed += (Pstart - P) * u1;
      acc.escaped += P * u1;
      return EV_DONE;
    }
    return EV_NONE;
  }
  static constexpr bool kStaged = false;
  __device__ __forceinline__ void begin_visit() {}
  // Budget of the parent's run when it splits (children carry P/4 each).
  __device__ __forceinline__ void on_split(const TraceArgs& A, LaneAcc& acc) const {
    acc.absorbed += (Pstart - P) * unit(A);
  }
  __device__ __forceinline__ void on_start_outside(const TraceArgs& A, LaneAcc& acc) const {
    acc.escaped += P * unit(A);
  }
};

// Optical depth that the FP64 evaluation accumulates along the lineage of
// package (level, pix) of source src up to and including its segment in cell
// (tc0, tc1, tc2).  Follows the FP64 path from the root: the root pixel at
// level0 is pix >> 2 (level - level0); at each split the lineage continues
// with the child on the path to pix.  If the lineage does not
// reach that cell at that level (returns NaN; the caller then keeps its FP32
// decision).
__device__ __forceinline__ double retrace_tau64(const TraceArgs& A, uint32_t src, int level, uint32_t pix, int tc0,
                                                int tc1, int tc2) {
  const SourceDev& S = A.src[src];
  const InstDev& I = A.inst[S.inst];
  const double s0 = S.s[0], s1 = S.s[1], s2 = S.s[2];
  int l = A.level0;
  double r = 0.0, tau = 0.0;
  for (int guard = 0; guard <= RT_MAX_LEVEL + 1; ++guard) {
    const uint32_t p = pix >> (2 * (level - l));
    double n[3];
    pix2vec64(l, p, n);
    int c0 = cell_of64(__dadd_rn(s0, __dmul_rn(r, n[0])), n[0]);
    int c1 = cell_of64(__dadd_rn(s1, __dmul_rn(r, n[1])), n[1]);
    int c2 = cell_of64(__dadd_rn(s2, __dmul_rn(r, n[2])), n[2]);
    double t0 = next_t64(c0, s0, n[0]), t1 = next_t64(c1, s1, n[1]), t2 = next_t64(c2, s2, n[2]);
    bool split = false;
    for (int st = 0; st < A.max_steps; ++st) {
      if (c0 < 0 || c0 >= I.nx || c1 < 0 || c1 >= I.ny || c2 < 0 || c2 >= I.nz) return nan("");
      const double rn = fmin(t0, fmin(t1, t2));
      if (l < A.max_level && rn > A.rsplit[l]) { split = true; break; }
      double dr = __dsub_rn(rn, r);
      if (dr < 0) dr = 0;
      const int idx = c0 + I.nx * (c1 + I.ny * c2);
      const double nh = S.type == 0 ? __dmul_rn(I.nH[idx], I.xHI[idx]) : I.nhe64[S.type - 1][idx];
      tau = __dadd_rn(tau, __dmul_rn(__dmul_rn(S.sdx, nh), dr));
      if (l == level && c0 == tc0 && c1 == tc1 && c2 == tc2) return tau;
      if (tau > A.tau_term) return nan("");
      if (n[0] != 0 && t0 == rn) { c0 += n[0] > 0 ? 1 : -1; t0 = next_t64(c0, s0, n[0]); }
      if (n[1] != 0 && t1 == rn) { c1 += n[1] > 0 ? 1 : -1; t1 = next_t64(c1, s1, n[1]); }
      if (n[2] != 0 && t2 == rn) { c2 += n[2] > 0 ? 1 : -1; t2 = next_t64(c2, s2, n[2]); }
      r = rn;
    }
    if (!split || l >= level) return nan("");
    ++l;
  }
  return nan("");
}

// ---------------------------------------------------------------------------
// FP32-mixed walker.
//
// All per-segment arithmetic is FP32.  Crossing distances t_i, the radius r,
// segment lengths and the optical depth are carried as unevaluated FP32 pairs
// (hi + lo, "double-float"), built from the pixel direction stored as an FP32
// pair (FP64 direction rounded twice) and from the source position as an FP32
// pair, so each t carries ~44 correct bits while every instruction is FP32.
// Attenuation and the k_ph / Gamma deposits are plain FP32.
//
// The walker is bound by its dependent instructions and the warps' issue
// slots (four warps per scheduler at 128 registers), so a segment's common
// case is kept short: planes are counted along each axis instead of located
// from cell indices (Axis), one comparison with a radius set at the package's
// start covers split, box exit and halt, one more the termination, and the
// decisions in full (decide, terminates) run only for a segment that fails
// either comparison or whose two nearest planes lie within 2^-20 of each
// other.  Source constants sit in registers; what only a package's end needs
// sits in shared memory.  With the decisions in full at every segment the
// trace of the 128^3 Stroemgren snapshot took 0.41 instead of 0.30 ms, 24 sources
// in an ionised 128^3 grid 13.2 instead of 9.6 ms, 1000 in a clumpy 256^3 grid 3.9
// instead of 3.3 ms; with the figures given at the steps below they take
// 0.23, 6.05 and 2.49 ms.
//
// Each decision that shapes the ray tree -- which cell plane is crossed next,
// whether the package splits, whether it terminates -- is taken from the
// FP32 values only when an error bound proves it equals the FP64 decision:
//   |t_pair - t_FP64| <= 2^-40 t + 2^-46 |s| / |n|   (per axis),
//   |tau_pair - tau_FP64| <= tau_bound (per package).
// Inside a band the decision is re-taken in FP64: the crossing distances of
// the current cell from the FP64 direction, or the FP64 optical depth of the
// package's lineage.  Per-level counts therefore equal the FP64 path's.
// ---------------------------------------------------------------------------
constexpr float kEps32 = 5.9604645e-8f;   // 2^-24
constexpr float kBandT = 9.094947e-13f;   // 2^-40
constexpr float kNear = 9.53674316e-7f;   // 2^-20: high parts farther apart are ordered

// Direction of a pixel of a level beyond the table, from the FP64 evaluation
// (out of line: its FP64 registers would otherwise press on every start).
struct DirPair {
  F2 n0, n1, n2;
  int diag;
};
__device__ __noinline__ DirPair dir_pair64(int level, uint32_t pix) {
  double v[3];
  DirPair d;
  d.diag = pix2vec64(level, pix, v);
  d.n0 = f2_from_double(v[0]);
  d.n1 = f2_from_double(v[1]);
  d.n2 = f2_from_double(v[2]);
  return d;
}

// Direction of (level, pix) as FP32 pairs: from the device table when the
// level is tabulated, else from the FP64 evaluation.  Returns the
// 45-degree-meridian flag.
__device__ __forceinline__ int dir_pair(const TraceArgs& A, int level, uint32_t pix, F2 n[3]) {
  if (level <= A.dir_levels) {
    const size_t idx = (size_t)4 * (((size_t)1 << (2 * level)) - 1) + pix;
    const float4 h = __ldg(&A.dir_tab[2 * idx]);
    const float4 l = __ldg(&A.dir_tab[2 * idx + 1]);
    n[0] = {h.x, l.x};
    n[1] = {h.y, l.y};
    n[2] = {h.z, l.z};
    return h.w != 0.0f;
  }
  const DirPair d = dir_pair64(level, pix);
  n[0] = d.n0;
  n[1] = d.n1;
  n[2] = d.n2;
  return d.diag;
}

// Exact (FP64) crossing decision for cell (c0, c1, c2) of package (level,
// pix) of source src: bit 3 = split, bits 0-2 = axes that reach the next
// plane first, among those of `near` (bits 0-2; the pairs prove the others
// later), bit 6 = the crossing lies beyond the halting radius rlim (+inf
// without a finite speed of light).  Inlined where it is used once: as a call it
// cost the kernel's caller-saved registers (28 spilled words).  The FP64
// direction is kept with the lane's sums: a ray whose planes nearly tie at every
// step (a source at x = 5.3, y = 60.3) asks for it as often, and with it formed
// and three quotients taken each time its trace took 0.27 ms in a neutral 128^3
// box and 0.95 in an ionised one, now 0.235 and 0.83.
__device__ __forceinline__ int decide64(const TraceArgs& A, LaneAcc& acc, uint32_t src, int level, uint32_t pix, int c0,
                                        int c1, int c2, int near, double rlim) {
  const SourceDev& S = A.src[src];
  if (acc.n_level != (uint32_t)level || acc.n_pix != pix) {
    double v[3];
    pix2vec64(level, pix, v);
    acc.n[0] = v[0]; acc.n[1] = v[1]; acc.n[2] = v[2];
    acc.n_level = (uint32_t)level;
    acc.n_pix = pix;
  }
  const double n[3] = {acc.n[0], acc.n[1], acc.n[2]};
  const double inf = __longlong_as_double(0x7ff0000000000000LL);
  const double u0 = near & 1 ? next_t64(c0, S.s[0], n[0]) : inf;
  const double u1 = near & 2 ? next_t64(c1, S.s[1], n[1]) : inf;
  const double u2 = near & 4 ? next_t64(c2, S.s[2], n[2]) : inf;
  const double rn = fmin(u0, fmin(u1, u2));
  int out = 0;
  if (level < A.max_level && rn > A.rsplit[level]) out |= 8;
  if (rn > rlim) out |= 64;
  if (n[0] != 0 && u0 == rn) out |= 1;
  if (n[1] != 0 && u1 == rn) out |= 2;
  if (n[2] != 0 && u2 == rn) out |= 4;
  return out;
}

// One axis of a ray.  Planes crossed by the axis are met at the distances
//   t = |plane - s| / |n|,  |plane - s| = d for a source on the 1/16-cell
// lattice (EXACT: d is an exact FP32 number and grows by exactly 1 per
// plane), else k + off |n| with k an integer and off the source's offset from
// the nearest integer, times 1 / |n|.  So the next plane of an axis costs
// four (EXACT) or ten FP32 instructions and no table or source record.  t is
// a pair whose low part may reach 2^-22 of the high part (it is not
// renormalised; every use allows for that).
constexpr float kFar = 1e30f;  // crossing distance of an axis that the ray never crosses
template <bool EXACT>
struct Axis {
  F2 iv;       // 1 / |n| (0 for a vanishing component)
  F2 t;        // distance to the next plane
  F2 off;      // general: offset term of t
  float d;     // EXACT
  int k;       // general
  int stride;  // change of the cell index at a plane (its sign is the direction's)
  __device__ __forceinline__ void plane() {
    const float f = EXACT ? d : (float)k;
    const float p = __fmul_rn(f, iv.hi);
    float e = fmaf(f, iv.hi, -p);
    e = fmaf(f, iv.lo, e);
    if (EXACT) {
      t = F2{p, e};
    } else {
      // k = 0, or |k| >= 1 and |off| <= iv / 2: the first sum's error is exact
      const float h = __fadd_rn(p, off.hi);
      const float z = __fadd_rn(__fsub_rn(p, h), off.hi);
      t = F2{h, __fadd_rn(__fadd_rn(e, z), off.lo)};
    }
  }
  __device__ __forceinline__ void next() {
    if (EXACT) d += 1.0f;
    else ++k;
    plane();
  }
  __device__ __forceinline__ void back() {
    if (EXACT) d -= 1.0f;
    else --k;
    plane();
  }
  // Cell c of an axis with direction n, source coordinate s (EXACT) or
  // sa + sb (general), dim cells and index stride `step`.
  __device__ __forceinline__ void init(int c, F2 n, float s, int sa, F2 sb, int step) {
    const bool neg = n.hi < 0.0f;
    iv = n.hi != 0.0f ? f2_recip(n) : F2{0.0f, 0.0f};
    if (neg) iv = F2{-iv.hi, -iv.lo};
    stride = n.hi > 0.0f ? step : (neg ? -step : 0);
    off = F2{0.0f, 0.0f};
    if (EXACT) {
      d = neg ? s - (float)c : (float)(c + 1) - s;
    } else {
      k = neg ? sa - c : c + 1 - sa;
      if (!neg) sb = F2{-sb.hi, -sb.lo};
      off = n.hi != 0.0f ? f2_mul(sb, iv) : sb;
    }
    if (n.hi != 0.0f) plane();
    else t = F2{kFar, 0.0f};
  }
  // the cell that init was given, advanced by the planes crossed since
  __device__ __forceinline__ int cell(float s, int sa) const {
    if (EXACT) return stride < 0 ? (int)(s - d) : (int)(s + d) - 1;
    return stride < 0 ? sa - k : sa + k - 1;
  }
  // direction cosine, for off_middle()
  __device__ __forceinline__ float cosine() const {
    const float n = iv.hi != 0.0f ? __frcp_rn(iv.hi) : 0.0f;
    return stride < 0 ? -n : n;
  }
  // distance along the axis (direction cosine n) of the point at radius rm from the middle of the cell
  __device__ __forceinline__ float off_middle(float n, float rm, float s, int sa) const {
    return fabsf(fmaf(n, rm, s) - ((float)cell(s, sa) + 0.5f));
  }
};

// EXACT: every source of the launch lies on the 1/16-cell lattice.  PAIR:
// n_HI is stored as FP32 pairs, and k_ph and Gamma side by side, so that a
// heating segment deposits both with one two-word reduction.  L2 takes those
// at the rate of single ones (200 G/s into 16 MB; two single ones 102 G/s):
// 24 sources in an ionised 128^3 grid 9.27 -> 8.45 ms, 30 of three photon types
// in 128^3 4.23 -> 3.89 ms, 1000 in a clumpy 256^3 grid 3.01 -> 2.92 ms.
// FC: deposits are scaled by the covering factor (its own instantiation,
// because its cell centres cost the segment loop 12 registers).
template <bool EXACT, bool PAIR, bool FC>
struct Walk32 {
  static constexpr bool kStaged = true;  // step() leaves rare decisions to slow() and terminate()
  using Rec = Rec32;  // packages in flight between traces; records of FSL traces
  template <bool FSL> using Q = typename std::conditional<FSL, Rec32, QRec32>::type;  // queue record
  uint32_t src, pix;
  uint32_t age;         // traces since emission (finite speed of light)
  F2 rlim;              // halting radius of this age
  uint32_t level;       // bits 0-3 level, bit 8: 45-degree ray whose x and y planes tie exactly
  F2 r;
  float P, tau, tau_lo;
  float tau_err;        // error bound of tau (in records and while a package starts or ends)
  Axis<EXACT> a0, a1, a2;
  int idx;              // cell index
  int cnt;              // segments of the package in this queue visit
  unsigned nseg;
  float nh, nh_lo;      // n_HI of the current cell (pair), loaded one step ahead
  float lim;            // below it no crossing splits, leaves the box or halts
  float sk, q;          // sum of kappa over the package's segments; error of tau per unit of it
  float sdx, sdx_lo, w, heat;
  float n0, n1, n2;     // FC: direction cosines
  const float* nhi;
  float* K;             // PAIR: (k_ph, Gamma) per cell
  float* G;             // else

  __device__ __forceinline__ int lvl() const { return (int)(level & 15u); }
  __device__ __forceinline__ bool diag_exact() const { return (level & 256u) != 0; }
  __device__ __forceinline__ void load_nh() {
    if (PAIR) {
      const float2 v = __ldg(reinterpret_cast<const float2*>(nhi) + idx);
      nh = v.x;
      nh_lo = v.y;
    } else {
      nh = __ldg(&nhi[idx]);
      nh_lo = 0.0f;
    }
  }
  // P of a new package of source S (finite speed of light)
  __device__ __forceinline__ double emit(const SourceDev& S) {
    P = __ldg(&S.sabs32.w);
    return (double)P;
  }
  __device__ __forceinline__ int inst(const TraceArgs& A) const { return A.src[src].inst; }
  __device__ __forceinline__ double unit(const TraceArgs& A) const { return A.src[src].unit; }
  // cell of coordinate u along an axis (tie rule: n > 0 floor, n < 0 ceil - 1)
  __device__ __forceinline__ static int cell_of(F2 u, float n) {
    const int f = f2_floor(u);
    if (n < 0.0f && (float)f == u.hi && u.lo == 0.0f) return f - 1;
    return f;
  }

  // A package at radius r: the absorber and accumulators of its photon type
  // (Sec. 3.2), its direction, first cell (the cell index `cell` when given:
  // a package continued from the previous trace; else the cell holding the
  // point at r), next crossings and limits.  False when that cell is outside
  // the box.
  template <bool FSL>
  __device__ __forceinline__ bool start(const TraceArgs& A, LaneAcc& acc, bool given, uint32_t cell) {
    const SourceDev& S = A.src[src];
    const InstDev& I = A.inst[A.ninst == 1 ? 0 : S.inst];  // (one dependent load less)
    const float4 sh = __ldg(&S.s32);
    const float4 sl = __ldg(&S.slo32);
    acc.Pstart = P;
    acc.tau0 = tau;
    acc.tau_err = tau_err;
    acc.steps = 0;
    cnt = 0;
    sk = 0.0f;
    F2 n[3];
    const int diag = dir_pair(A, lvl(), pix, n);
    const int ties = (n[0].hi < 0.0f) == (n[1].hi < 0.0f) ? 1 : 2;
    level = (level & 15u) | ((diag && ((int)sh.w & ties)) ? 256u : 0u);
    const int nx = I.nx, ny = I.ny, nz = I.nz;
    int c0, c1, c2;
    if (FSL && given) {
      c0 = (int)(cell % (uint32_t)nx);
      c1 = (int)((cell / (uint32_t)nx) % (uint32_t)ny);
      c2 = (int)(cell / ((uint32_t)nx * (uint32_t)ny));
    } else {
      // the point in FP32 where that is clear of every plane by more than its
      // error, else as pairs
      const float u0 = fmaf(r.hi, n[0].hi, sh.x), u1 = fmaf(r.hi, n[1].hi, sh.y), u2 = fmaf(r.hi, n[2].hi, sh.z);
      const float f0 = floorf(u0), f1 = floorf(u1), f2 = floorf(u2);
      const float far = fmaxf(fabsf(u0 - f0 - 0.5f), fmaxf(fabsf(u1 - f1 - 0.5f), fabsf(u2 - f2 - 0.5f)));
      if (far < 0.5f - 8.0f * kEps32 * (r.hi + fmaxf(sh.x, fmaxf(sh.y, sh.z)))) {
        c0 = (int)f0;
        c1 = (int)f1;
        c2 = (int)f2;
      } else {
        c0 = cell_of(f2_add(F2{sh.x, sl.x}, f2_mul(r, n[0])), n[0].hi);
        c1 = cell_of(f2_add(F2{sh.y, sl.y}, f2_mul(r, n[1])), n[1].hi);
        c2 = cell_of(f2_add(F2{sh.z, sl.z}, f2_mul(r, n[2])), n[2].hi);
      }
      if (c0 < 0 || c0 >= nx || c1 < 0 || c1 >= ny || c2 < 0 || c2 >= nz) return false;
    }
    idx = c0 + nx * (c1 + ny * c2);
    const int t = S.type;
    nhi = (const float*)(t == 0 ? I.nhi : I.nhe[t - 1]);
    load_nh();
    if (EXACT) {
      a0.init(c0, n[0], sh.x, 0, F2{0.0f, 0.0f}, 1);
      a1.init(c1, n[1], sh.y, 0, F2{0.0f, 0.0f}, nx);
      a2.init(c2, n[2], sh.z, 0, F2{0.0f, 0.0f}, nx * ny);
    } else {
      const float4 bh = __ldg(&S.sb32), bl = __ldg(&S.sblo32);
      a0.init(c0, n[0], sh.x, S.sa[0], F2{bh.x, bl.x}, 1);
      a1.init(c1, n[1], sh.y, S.sa[1], F2{bh.y, bl.y}, nx);
      a2.init(c2, n[2], sh.z, S.sa[2], F2{bh.z, bl.z}, nx * ny);
    }
    if (FC) {
      n0 = a0.cosine();
      n1 = a1.cosine();
      n2 = a2.cosine();
    }
    K = (float*)(t == 0 ? I.K : I.Khe[t - 1]);
    if (!PAIR) G = (float*)I.G;
    const float4 k32 = __ldg(&S.k32);  // sdx, w, rw, heat
    sdx = k32.x; sdx_lo = sl.w; w = k32.y; heat = k32.w;
    // The radius below which no crossing splits, leaves the box or halts: the
    // exit plane of each axis (its distance from the source in FP32, less the
    // rounding of s and of the product), the split and the halting radius;
    // and a bound on the radius for the error of tau.
    float lo = exit_of(a0, n[0].hi < 0.0f ? sh.x : (float)nx - sh.x, (float)nx);
    lo = fminf(lo, exit_of(a1, n[1].hi < 0.0f ? sh.y : (float)ny - sh.y, (float)ny));
    lo = fminf(lo, exit_of(a2, n[2].hi < 0.0f ? sh.z : (float)nz - sh.z, (float)nz));
    float hi = (float)nx + (float)ny + (float)nz;
    const int l = lvl();
    if (l < A.max_level) {
      lo = fminf(lo, A.rsplit32[l]);
      hi = fminf(hi, A.rsplit32[l]);
    }
    if (FSL) lo = fminf(lo, rlim.hi);
    acc.lim = fmaf(lo, -kNear, lo);
    lim = r.hi == 0.0f ? 0.0f : acc.lim;  // segments from the source itself: slow(), with deposit_first()
    const float4 sa = __ldg(&S.sabs32);
    q = fmaf(hi, 4.1f * kBandT, 1e-30f) +
        4.1f * fmaxf(sa.x * a0.iv.hi, fmaxf(sa.y * a1.iv.hi, sa.z * a2.iv.hi));
    // step() compares tau + sk q with tau_near, 2^-12 below the termination.
    // Beside its own boundaries (sk q) a package's error comes from the pair
    // products (2^-37 of tau; 2^-22 where n_HI is plain FP32), from the sums
    // (2^-18 at most over the 24,600 planes of a 4096^3 grid), and from its
    // ancestors, which clip dense cells over lengths that are hardly known:
    // where those leave more than half of the 2^-12, every segment takes the
    // full test.
    if (!(tau_err <= A.tau_term32 * (1.0f / 8192.0f))) q = 1e30f;
    return true;
  }
  __device__ __forceinline__ static float exit_of(const Axis<EXACT>& a, float d, float dim) {
    return a.iv.hi > 0.0f ? fmaf(dim, -8.0f * kEps32, d) * a.iv.hi : kFar;
  }
  __device__ __forceinline__ void set_rlim(const TraceArgs& A) {
    if ((int)age < A.n_ages) {
      const float2 v = __ldg(&A.rlim32[age]);
      rlim = F2{v.x, v.y};
    } else {
      set_status(A.ctl, RT_ERR_STATE);
      rlim = F2{0.0f, 0.0f};
    }
  }

  __device__ __forceinline__ void load(const Rec& q_) {
    r = {q_.r, q_.r_lo}; P = q_.P; tau = q_.tau; tau_lo = q_.tau_lo; tau_err = q_.tau_err; src = q_.src; pix = q_.pix;
    level = q_.tag & 15u;
    age = q_.age;
  }
  // Bound on |tau (pair) - tau (FP64 evaluation)| at radius rmax.  Each
  // crossing's pair lies within 2^-40 t + 2^-46 |s| / |n| of the FP64 one and
  // shifts the boundary between two cells, so tau by at most that times the
  // two kappas (twice that, with margin); the pair products add 2^-37 dtau
  // (2^-22 dtau where n_HI is plain FP32), and the pair sum 2^-44 tau a
  // segment plus the rounding of its low part, which is renormalised once per
  // queue visit and so stays below segs_per_iter 2^-24 tau.
  __device__ __forceinline__ float tau_bound(const TraceArgs& A, const LaneAcc& acc, float rmax) const {
    const float4 sa = __ldg(&A.src[src].sabs32);
    const float ab = fmaxf(sa.x * a0.iv.hi, fmaxf(sa.y * a1.iv.hi, sa.z * a2.iv.hi));
    const float e_dtau = PAIR ? 8.0f * kBandT : 4.0f * kEps32;
    const float spi = (float)A.segs_per_iter;
    return acc.tau_err + fmaf(tau, kEps32, tau - acc.tau0) * e_dtau + sk * (fmaf(rmax, 4.0f * kBandT, 1e-30f) + 4.0f * ab) +
           (float)(acc.steps + cnt) * tau * (kBandT / 16.0f + spi * (kEps32 * kEps32));
  }
  // The package's radius and optical depth as normalised pairs with the error
  // bound, for its children or the store of packages in flight.
  __device__ __forceinline__ void seal(const TraceArgs& A, const LaneAcc& acc) {
    r = fast_two_sum(r.hi, r.lo);
    const F2 t2 = fast_two_sum(tau, tau_lo);
    tau = t2.hi;
    tau_lo = t2.lo;
    tau_err = tau_bound(A, acc, r.hi);
  }
  // Record of child cpix (level + 1, P/4, same radius, age, optical depth and
  // its error bound); the level sits in the tag's low bits until publication.
  __device__ __forceinline__ Rec make_child(uint32_t cpix) const {
    Rec c;
    c.r = r.hi; c.r_lo = r.lo; c.P = P * 0.25f; c.tau = tau; c.tau_lo = tau_lo; c.tau_err = tau_err;
    c.src = src; c.pix = cpix; c.tag = (uint32_t)(lvl() + 1); c.age = age;
    return c;
  }
  __device__ __forceinline__ static uint32_t cell_of_record(const Rec& q_) { return q_.cell; }
  // A halted package as the next trace continues it (one trace older).
  __device__ __forceinline__ void store_halted(Rec* q_) const {
    reinterpret_cast<float4*>(&q_->r)[0] = make_float4(r.hi, r.lo, P, tau);
    reinterpret_cast<uint4*>(&q_->tau_lo)[0] =
        make_uint4(__float_as_uint(tau_lo), __float_as_uint(tau_err), src, pix);
    reinterpret_cast<uint4*>(&q_->tag)[0] = make_uint4((uint32_t)lvl(), age + 1, (uint32_t)idx, 0u);
  }
  // A record's payload into its queue slot; the tag that completes it follows
  // a fence.  FSL records (48 B) carry the age and the tag ((epoch << 4) |
  // level); the others (32 B) the level beside the source index and the tag
  // ((epoch & 0xffff) << 16 | tau_err as bf16 rounded up).
  template <bool FSL>
  __device__ __forceinline__ static void put(Q<FSL>* q, const Rec& c) {
    __stcg(reinterpret_cast<float4*>(&q->r), make_float4(c.r, c.r_lo, c.P, c.tau));
    if constexpr (FSL) {
      __stcg(reinterpret_cast<uint4*>(&q->tau_lo),
             make_uint4(__float_as_uint(c.tau_lo), __float_as_uint(c.tau_err), c.src, c.pix));
      __stcg(&q->age, c.age);
    } else {
      __stcg(reinterpret_cast<uint2*>(&q->tau_lo), make_uint2(__float_as_uint(c.tau_lo), c.src | ((c.tag & 15u) << 28)));
      __stcg(&q->pix, c.pix);
    }
  }
  template <bool FSL>
  __device__ __forceinline__ static uint32_t tag_of(const Rec& c, uint32_t epoch) {
    if constexpr (FSL) return (epoch << 4) | (c.tag & 15u);
    // tau_err >= 0: adding 0xffff before the shift rounds the magnitude up
    return (epoch << 16) | ((__float_as_uint(c.tau_err) + 0xffffu) >> 16);
  }
  // Poll with an acquire load of the tag: the payload reads that follow a
  // successful poll are ordered after it without a fence.
  template <bool FSL>
  __device__ __forceinline__ static bool poll(const Q<FSL>* q, uint32_t epoch, Rec& o) {
    const uint32_t tg = ld_acquire_u32(&q->tag);
    if constexpr (FSL) {
      if ((tg >> 4) != (epoch & 0x0fffffffu)) return false;
    } else {
      if ((tg >> 16) != (epoch & (uint32_t)kEpochMask)) return false;
    }
    const float4 a = __ldcg(reinterpret_cast<const float4*>(&q->r));
    const uint4 b = __ldcg(reinterpret_cast<const uint4*>(&q->tau_lo));
    o.r = a.x; o.r_lo = a.y; o.P = a.z; o.tau = a.w;
    o.tau_lo = __uint_as_float(b.x);
    if constexpr (FSL) {
      o.tau_err = __uint_as_float(b.y); o.src = b.z; o.pix = b.w; o.tag = tg;
      o.age = __ldcg(&q->age);
    } else {
      o.src = b.y & (kMaxQueueSources - 1u); o.tag = b.y >> 28; o.pix = b.z;
      o.tau_err = __uint_as_float(tg << 16);
      o.age = 0u;
    }
    return true;
  }
  // Every lane takes the record that lane `from` holds (all lanes call it).
  __device__ __forceinline__ static void shfl_rec(Rec& c, int from) {
    c.r = __shfl_sync(0xffffffffu, c.r, from);
    c.r_lo = __shfl_sync(0xffffffffu, c.r_lo, from);
    c.P = __shfl_sync(0xffffffffu, c.P, from);
    c.tau = __shfl_sync(0xffffffffu, c.tau, from);
    c.tau_lo = __shfl_sync(0xffffffffu, c.tau_lo, from);
    c.tau_err = __shfl_sync(0xffffffffu, c.tau_err, from);
    c.src = __shfl_sync(0xffffffffu, c.src, from);
    c.pix = __shfl_sync(0xffffffffu, c.pix, from);
    c.tag = __shfl_sync(0xffffffffu, c.tag, from);
    c.age = __shfl_sync(0xffffffffu, c.age, from);
  }
  __device__ __forceinline__ static Rec root_rec(uint32_t gsrc, uint32_t l, uint32_t p) {
    Rec c;
    c.r = 0.0f; c.r_lo = 0.0f; c.P = 1.0f; c.tau = 0.0f; c.tau_lo = 0.0f; c.tau_err = 0.0f; c.src = gsrc; c.pix = p;
    c.tag = l;
    c.age = 0u;
    return c;
  }
  __device__ __forceinline__ void become_child0() {
    level = (uint32_t)(lvl() + 1); pix = 4u * pix; P = P * 0.25f;
  }

  // The next crossing as the FP64 evaluation takes it, where the fast test of
  // step() cannot tell: bits 0-2 the planes crossed, bit 3 a split first, bit
  // 6 (FSL) the crossing lies beyond the halting radius, bit 7 the crossing
  // leaves the box; rn receives the crossing distance.  Orders that the pairs
  // cannot prove are re-taken in FP64 (decide64) and counted in fb.
  template <bool FSL>
  __device__ __forceinline__ int decide(const TraceArgs& A, LaneAcc& acc, F2& rn, unsigned& fb) const {
    const SourceDev& S = A.src[src];
    int imin = 0;
    rn = a0.t;
    if (f2_diff(a1.t, rn) < 0.0f) { rn = a1.t; imin = 1; }
    if (f2_diff(a2.t, rn) < 0.0f) { rn = a2.t; imin = 2; }
    const float4 sab = __ldg(&S.sabs32);
    const float b0 = fmaf(a0.t.hi, kBandT, sab.x * a0.iv.hi), b1 = fmaf(a1.t.hi, kBandT, sab.y * a1.iv.hi),
                b2 = fmaf(a2.t.hi, kBandT, sab.z * a2.iv.hi);
    const float emin = imin == 0 ? b0 : (imin == 1 ? b1 : b2);
    bool m0 = imin == 0, m1 = imin == 1, m2 = imin == 2;
    bool unsure = false;
    int near = 1 << imin;  // the axes among which the pairs leave the first plane open
    const bool xy_tie = diag_exact();  // planes this close are an exact tie then (see step)
    if (!m0 && f2_diff(a0.t, rn) <= b0 + emin) { near |= 1; if (imin == 1 && xy_tie) m0 = true; else unsure = true; }
    if (!m1 && f2_diff(a1.t, rn) <= b1 + emin) { near |= 2; if (imin == 0 && xy_tie) m1 = true; else unsure = true; }
    if (!m2 && f2_diff(a2.t, rn) <= b2 + emin) { near |= 4; unsure = true; }
    const int l = lvl();
    bool split = false, halt = false;
    if (l < A.max_level) {
      const float R = A.rsplit32[l];
      const float d = f2_diff(rn, F2{R, A.rsplit32lo[l]});
      split = d > 0.0f;
      if (fabsf(d) <= emin + R * kBandT) unsure = true;
    }
    if (FSL) {  // Step 3j: the crossing against the halting radius, decided like the split
      const float d = f2_diff(rn, rlim);
      halt = d > 0.0f;
      if (fabsf(d) <= emin + rlim.hi * kBandT) unsure = true;
    }
    const float4 sh = __ldg(&S.s32);
    const int c0 = a0.cell(sh.x, S.sa[0]), c1 = a1.cell(sh.y, S.sa[1]), c2 = a2.cell(sh.z, S.sa[2]);
    if (unsure) {
      const double rlim64 = !FSL ? __longlong_as_double(0x7ff0000000000000LL)
                                 : ((int)age < A.n_ages ? A.rlim64[age] : 0.0);
      const int d64 = decide64(A, acc, src, l, pix, c0, c1, c2, near, rlim64);
      split = (d64 & 8) != 0;
      halt = (d64 & 64) != 0;
      m0 = (d64 & 1) != 0;
      m1 = (d64 & 2) != 0;
      m2 = (d64 & 4) != 0;
      ++fb;
    }
    const InstDev& I = A.inst[S.inst];
    const bool out = (m0 && (a0.stride < 0 ? c0 == 0 : c0 + 1 == I.nx)) ||
                     (m1 && (a1.stride < 0 ? c1 == 0 : c1 + 1 == I.ny)) ||
                     (m2 && (a2.stride < 0 ? c2 == 0 : c2 + 1 == I.nz));
    return (m0 ? 1 : 0) | (m1 ? 2 : 0) | (m2 ? 4 : 0) | (split ? 8 : 0) | (halt ? 64 : 0) | (out ? 128 : 0);
  }

  // The segment from r to `end` in a cell of density (nh, nh_lo); returns its k_ph.
  __device__ __forceinline__ float segment(const TraceArgs& A, LaneAcc& acc, F2 r, F2 end, float nh, float nh_lo) {
    // length as a pair (both ends are pairs; |end| >= |r| or the difference of
    // the high parts is exact)
    const float dh = __fsub_rn(end.hi, r.hi);
    const float dl = __fadd_rn(__fsub_rn(__fsub_rn(end.hi, dh), r.hi), __fsub_rn(end.lo, r.lo));
    float dr = __fadd_rn(dh, dl);
    float drl = __fadd_rn(__fsub_rn(dh, dr), dl);
    ++cnt;
    if (!(dr > 0.0f)) {  // a start on a plane, a tie: no length, not counted
      dr = 0.0f;
      drl = 0.0f;
      --nseg;
    }
    // kappa = sigma dx n_HI and dtau = kappa dr as pairs: the optical depth
    // follows the FP64 sum to ~2^-44 where n_HI is a pair
    const float kap = __fmul_rn(sdx, nh);
    float kl = fmaf(sdx, nh, -kap);
    if (PAIR) kl = fmaf(sdx, nh_lo, kl);
    kl = fmaf(sdx_lo, nh, kl);
    const float dp = __fmul_rn(kap, dr);
    float de = fmaf(kap, dr, -dp);
    de = fmaf(kap, drl, de);
    de = fmaf(kl, dr, de);
    const float dtau = __fadd_rn(dp, de);
    const float dtl = __fadd_rn(__fsub_rn(dp, dtau), de);
    // transmitted fraction tr = e^-tau; phi = (1 - e^-tau)/tau from its Taylor
    // series below tau = 1/4 (7 terms: the first dropped term, tau^7 / 8!, is
    // below 1.6e-9 there, under FP32 rounding), else from tr.
    // Both are computed and one is selected, so lanes do not diverge.
    const float tr = expf(-dtau);
    const float ser = fmaf(fmaf(fmaf(fmaf(fmaf(fmaf(dtau, 1.0f / 5040.0f, -1.0f / 720.0f), dtau, 1.0f / 120.0f), dtau,
                                          -1.0f / 24.0f), dtau, 1.0f / 6.0f), dtau, -0.5f), dtau, 1.0f);
    const float phi = dtau < 0.25f ? ser : __fdividef(1.0f - tr, dtau);
    float fcv = 1.0f;
    if (FC) {
      fcv = cover(A, r, dr);
      acc.cover = fcv;
    }
    const float k = P * w * dr * phi * fcv;
    P = P * tr;
    // the larger summand first: the sum's rounding error is exact
    const float s = __fadd_rn(tau, dtau);
    const float e = __fsub_rn(fminf(tau, dtau), __fsub_rn(s, fmaxf(tau, dtau)));
    tau_lo = __fadd_rn(tau_lo, __fadd_rn(e, dtl));
    tau = s;
    sk += kap;
    return k;
  }
  // covering factor (Eq. "fc") of a segment of length dr, in FP32 from the
  // pairs' high parts: its error (~1e-4 relative) is far inside the tolerance
  // on k_ph
  __device__ __forceinline__ float cover(const TraceArgs& A, F2 r, float dr) const {
    const float rh = __fadd_rn(r.hi, r.lo);
    const float L = rh * A.theta32[lvl()];
    if (!(L > 0.0f)) return 1.0f;
    const float4 sh = __ldg(&A.src[src].s32);
    const int* sa = A.src[src].sa;
    const float rm = fmaf(0.5f, dr, rh);
    const float d = fmaxf(a0.off_middle(n0, rm, sh.x, sa[0]), fmaxf(a1.off_middle(n1, rm, sh.y, sa[1]), a2.off_middle(n2, rm, sh.z, sa[2])));
    const float f = 0.5f + (0.5f - d) / L;
    return fminf(1.0f, f * f);
  }
  // Cross the planes m0, m1, m2 at rn; the next cell's density is loaded a
  // step ahead.
  __device__ __forceinline__ void advance(F2 rn, bool m0, bool m1, bool m2) {
    enter(m0, m1, m2);
    cross(rn, m0, m1, m2);
  }
  __device__ __forceinline__ void enter(bool m0, bool m1, bool m2) {
    if (m0) idx += a0.stride;
    if (m1) idx += a1.stride;
    if (m2) idx += a2.stride;
    load_nh();
  }
  __device__ __forceinline__ void cross(F2 rn, bool m0, bool m1, bool m2) {
    r = rn;
    if (m0) a0.next();
    if (m1) a1.next();
    if (m2) a2.next();
  }

  // One segment of the common case.  EV_RARE leaves the package before a
  // segment that may split, leave the box or halt, or whose next plane is not
  // provably the nearest; EV_TERM after one that may end it.
  template <bool FSL>
  __device__ __forceinline__ int step(const TraceArgs& A, LaneAcc& acc) {
    // The next plane: the smallest high part, provably the nearest when no
    // other is within 2^-20 of it (each is within 2^-22 of its distance).
    F2 rn;
    rn.hi = fminf(a0.t.hi, fminf(a1.t.hi, a2.t.hi));
    const float close = fmaf(rn.hi, kNear, rn.hi);
    const bool m0 = a0.t.hi <= close, m1 = a1.t.hi <= close, m2 = a2.t.hi <= close;
    rn.lo = m0 ? a0.t.lo : (m1 ? a1.t.lo : a2.t.lo);
    if (rn.hi >= lim || (m2 && (m0 || m1))) return EV_RARE;
    // The exact tie of a 45-degree ray crosses both planes: where its x and y
    // planes tie (fill_position32), planes within 2^-20 of each other are equal.
    // (Equal pairs were asked for before, which the general form, whose offsets
    // round either way, does not always give, and a source on the 1/16-cell
    // lattice: an FP64 decision at every other tie, which ends the lane's visit.
    // In the allocation-free trace of 30 sources in 48^3 cells 1875 of them, 242 us
    // instead of 171; the trace from a source at a third of a neutral 128^3 box
    // 0.28 ms instead of 0.09, of an ionised one 1.13 instead of 0.40.)
    if (m0 && m1) {
      if (!diag_exact()) return EV_RARE;
      if (!EXACT) rn.hi = a0.t.hi;  // one distance in two pairs: high and low part of the same one
    }
    // cross first: the next cell's density arrives while this segment's
    // absorption is worked out (24 sources in an ionised 128^3 grid 7.30 -> 6.81
    // ms).  With a covering factor the planes stay until it has read the cell
    // from them (with the whole crossing after the absorption, and the cosines
    // formed again in every segment: 1000 sources in a clumpy 256^3 grid 3.70
    // instead of 2.95 ms, 60 in 96^3 0.106 instead of 0.095 ms).
    const int at = idx;
    const F2 r0 = r;
    const float nh0 = nh, nh0_lo = nh_lo;
    if (FC) enter(m0, m1, m2);
    else advance(rn, m0, m1, m2);
    deposit(at, segment(A, acc, r0, rn, nh0, nh0_lo));
    if (FC) cross(rn, m0, m1, m2);
    if (fmaf(sk, q, tau) > A.tau_near) {
      // back to the cell (terminate() decides, and crosses again)
      if (m0) a0.back();
      if (m1) a1.back();
      if (m2) a2.back();
      idx = at;
      nh = nh0;
      nh_lo = nh0_lo;
      acc.mask = (m0 ? 1 : 0) | (m1 ? 2 : 0) | (m2 ? 4 : 0);
      return EV_TERM;
    }
    return EV_NONE;
  }

  // The segment that step() left at EV_RARE, with the full decision; its
  // k_ph in dep.  EV_TERM as in step(), bits 6 and 7 of acc.mask as from decide().
  template <bool FSL>
  __device__ __forceinline__ int slow(const TraceArgs& A, LaneAcc& acc, float& dep) {
    lim = acc.lim;
    F2 rn;
    unsigned fb = 0;
    const int m = decide<FSL>(A, acc, rn, fb);
    acc.fallbacks += fb;
    if (m & 8) return EV_SPLIT;
    const bool halt = FSL && (m & 64);  // Step 3j: the segment ends at rlim
    dep = segment(A, acc, r, halt ? rlim : rn, nh, nh_lo);
    acc.mask = m;
    if (fmaf(sk, q, tau) > A.tau_near) {
      r = rn;
      return EV_TERM;
    }
    return pass<FSL>(A, acc, rn);
  }
  // Past a segment that did not end the package by its optical depth: halted,
  // out of the box, or in the next cell.
  template <bool FSL>
  __device__ __forceinline__ int pass(const TraceArgs& A, LaneAcc& acc, F2 rn) {
    const int m = acc.mask;
    if (FSL && (m & 64)) {
      r = rlim;
      const double u = unit(A);
      acc.absorbed += ((double)acc.Pstart - (double)P) * u;
      acc.halted += (double)P * u;
      return EV_HALT;
    }
    if (m & 128) {
      leave(A, acc);
      return EV_DONE;
    }
    advance(rn, (m & 1) != 0, (m & 2) != 0, (m & 4) != 0);
    return EV_NONE;
  }
  // A segment left at EV_TERM: whether the package ends here (Step 3i), its
  // residual then added to dep.
  template <bool FSL>
  __device__ __forceinline__ int terminate(const TraceArgs& A, LaneAcc& acc, float& dep) {
    const bool halt = FSL && (acc.mask & 64);
    const float d = f2_diff(F2{tau, tau_lo}, F2{A.tau_term32, A.tau_term32lo});
    const float bnd = tau_bound(A, acc, r.hi) + tau * (4.0f * kBandT) + 1e-30f;
    bool term = d > bnd;
    if (!term && !(-d > bnd)) {
      // too close to call: the lineage's optical depth in FP64 (a lineage
      // emitted in an earlier trace crossed other media, and a cut segment
      // is not the cell's: there the pair's own decision stands)
      acc.fallbacks_tau++;
      double t64 = __longlong_as_double(0x7ff8000000000000LL);
      if (!FSL || (age == 0 && !halt)) {
        const SourceDev& S = A.src[src];
        const float4 sh = __ldg(&S.s32);
        t64 = retrace_tau64(A, src, lvl(), pix, a0.cell(sh.x, S.sa[0]), a1.cell(sh.y, S.sa[1]), a2.cell(sh.z, S.sa[2]));
      }
      term = isnan(t64) ? (d > 0.0f) : (t64 > A.tau_term);
    }
    if (!term) return pass<FSL>(A, acc, r);
    if (nh > 0.0f) dep += P * __ldg(&A.src[src].k32.z) / nh * (FC ? acc.cover : 1.0f);
    acc.absorbed += (double)acc.Pstart * unit(A);
    return EV_DONE;
  }
  // k into k_ph of cell `at`, k heat into its Gamma
  __device__ __forceinline__ void deposit(int at, float k) const {
    if (PAIR) {
      float* const p = K + 2 * (size_t)(unsigned)at;
      if (heat != 0.0f) red_add2(p, k, k * heat);
      else red_add(p, k);
    } else {
      red_add(&K[at], k);
      if (heat != 0.0f) red_add(&G[at], k * heat);
    }
  }
  // The same for segments that start at the source itself (the lanes with
  // `first`; every lane of the warp calls it).  The roots of a source land in
  // one cell (those of a source on a cell face in a few), its brightest, with
  // few distinct values whose FP32 sum rounds the same way again and again
  // (up to 2.6e-6 of the cell's rate); the lanes' shares are added as a pair
  // first, one reduction per cell and warp.
  __device__ __forceinline__ void deposit_first(bool first, int at, float k) const {
    const unsigned all = __ballot_sync(kFull, first);
    const unsigned mine = __match_any_sync(kFull, src) & __match_any_sync(kFull, at) & all;
    F2 s = {0.0f, 0.0f};
    for (unsigned m = all; m; m &= m - 1u) {
      const int l = __ffs(m) - 1;
      const float v = __shfl_sync(kFull, k, l);
      if ((mine >> l) & 1u) {
        const F2 t = two_sum(s.hi, v);
        s = F2{t.hi, __fadd_rn(s.lo, t.lo)};
      }
    }
    if (first && (int)(threadIdx.x & 31u) == __ffs(mine) - 1) deposit(at, __fadd_rn(s.hi, s.lo));
  }
  __device__ __forceinline__ void leave(const TraceArgs& A, LaneAcc& acc) const {
    const double u = unit(A);
    acc.absorbed += ((double)acc.Pstart - (double)P) * u;
    acc.escaped += (double)P * u;
  }
  // Around the segments of a queue visit: the pair sum renormalised before;
  // the segments counted, and their number bounded, after.
  __device__ __forceinline__ void begin_visit() {
    const F2 t2 = fast_two_sum(tau, tau_lo);
    tau = t2.hi;
    tau_lo = t2.lo;
  }
  __device__ __forceinline__ int end_visit(const TraceArgs& A, LaneAcc& acc, int ev) {
    nseg += cnt;
    acc.steps += cnt;
    cnt = 0;
    if (ev == EV_NONE && acc.steps > A.max_steps) {
      set_status(A.ctl, RT_ERR_STATE);
      leave(A, acc);
      return EV_DONE;
    }
    if (ev == EV_SPLIT || ev == EV_HALT) seal(A, acc);
    return ev;
  }
  __device__ __forceinline__ void on_split(const TraceArgs& A, LaneAcc& acc) const {
    acc.absorbed += ((double)acc.Pstart - (double)P) * unit(A);
  }
  __device__ __forceinline__ void on_start_outside(const TraceArgs& A, LaneAcc& acc) const {
    acc.escaped += (double)P * unit(A);
  }
};

// ---------------------------------------------------------------------------
// The persistent kernel, generic over the walker.
// ---------------------------------------------------------------------------
template <class W, int MinBlocks, bool FSL>
__global__ void __launch_bounds__(kBlock, MinBlocks) trace_kernel(TraceArgs A) {
  using Rec = typename W::Rec;
  __shared__ unsigned int sh_cnt[kShInst * kLevels];
  __shared__ unsigned long long sh_hsh[kShInst * kLevels];
  __shared__ LaneAcc sh_acc[kBlock];
  __shared__ unsigned int sh_bfb[kShInst * 2];
  __shared__ IdleWarp sh_idle[kBlock / 32];
  __shared__ uint32_t sh_epoch;
  for (int i = threadIdx.x; i < kShInst * kLevels; i += blockDim.x) {
    sh_cnt[i] = 0;
    sh_hsh[i] = 0;
  }
  double* const brow = A.blk + (size_t)blockIdx.x * A.blk_rows * kBlkRow;
  for (int i = threadIdx.x; i < A.blk_rows * kBlkRow; i += blockDim.x) brow[i] = 0.0;  // also 0 as an integer
  for (int i = threadIdx.x; i < kShInst * 2; i += blockDim.x) sh_bfb[i] = 0u;
  const BlockBudget BB{brow, A.blk_rows, sh_bfb};
  LaneAcc& acc = sh_acc[threadIdx.x];
  acc.emitted = acc.absorbed = acc.escaped = acc.resumed = acc.halted = 0.0;
  acc.segments = acc.fallbacks = acc.fallbacks_tau = 0;
  acc.inst = -1;
  acc.n_level = 0xffffffffu;
  if ((threadIdx.x & 31) == 0) sh_idle[threadIdx.x >> 5] = IdleWarp{-1, 0, 256u};
  if (threadIdx.x == 0) sh_epoch = (uint32_t)A.ctl[CTL_EPOCH];
  __syncthreads();
  LevelCounters LC{sh_cnt, sh_hsh};

  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  using QR = typename W::template Q<FSL>;
  QR* queue = (QR*)A.queue;
  // tickets: roots [0, n_roots), packages in flight [n_roots, qbase), queue slots after
  unsigned long long res_a = 0, n_res = 0;
  if (FSL) {
    res_a = A.ctl[CTL_RES_A];
    n_res = A.ctl[CTL_RES_B] - res_a;
  }
  const unsigned long long qbase = A.n_roots + n_res;

  W w;
  w.nseg = 0;
  bool active = false;
  int ev = EV_NONE;
  long long ticket = -1;
  IdleWarp& idle = sh_idle[threadIdx.x >> 5];

  for (;;) {
    // (1) What the last queue visit ended.  A split keeps child 0 and hands
    //     children 1-3 first to lanes of this warp that are free (no package
    //     and no ticket: in practice the lanes whose package ended in this
    //     round; a lane holding a ticket must stay free to take up the record
    //     that the ticket names), the rest to the queue (slots reserved
    //     together); finished packages leave the outstanding count, and the
    //     free lanes that get no child take a ticket.  Child j = 3 i + k - 1 of
    //     the i-th splitting lane goes to the j-th free lane when there is
    //     one, else to slot base + j - nin.
    //     One atomic per warp and counter (the count carries +3 per split, -1
    //     per finished package), all in flight together: a round waits for
    //     one trip to L2 where one after the other they took up to two, and
    //     for none of the count where nothing splits (with the shorter sleeps
    //     below: 128^3 Stroemgren snapshot 0.241 -> 0.232 ms, 24-grid batch 1.785
    //     -> 1.767 ms, 8 small grids 0.180 -> 0.173 ms).
    Start fresh = NO_START;  // a package starts in this lane now
    const bool split = (ev == EV_SPLIT);
    const bool done = ev == EV_DONE;
    const unsigned sm = __ballot_sync(kFull, split);
    const unsigned dm = __ballot_sync(kFull, done);
    const unsigned fm = __ballot_sync(kFull, !split && (!active || done) && ticket < 0);
    if (sm | dm | fm) {
      const unsigned nsp = __popc(sm);
      const unsigned nfree = __popc(fm);
      // (no hand-off in the finite-speed-of-light kernel, which spills at the
      // register cap already: there that code cost more than it saved)
      const unsigned nin = FSL ? 0u : (nfree < 3u * nsp ? nfree : 3u * nsp);  // children placed in this warp
      const unsigned nq = 3u * nsp - nin;                                   // children through the queue
      unsigned long long base = 0, tick = 0;
      if (lane == 0) {
        if (nfree > nin) tick = atomicAdd(&A.ctl[CTL_HEAD], (unsigned long long)(nfree - nin));
        const unsigned long long delta = (unsigned long long)(3LL * nsp - (long long)__popc(dm));
        if (sm) {
          // The count must include the children before any child is published,
          // or a consumer could finish a child and see it reach zero: wait for
          // the atomic's return value; the publishing lanes' fence follows.
          if (nq) base = atomicAdd(&A.ctl[CTL_TAIL], (unsigned long long)nq);
          const unsigned long long o = atomicAdd(&A.ctl[CTL_OUTSTANDING], delta);
          asm volatile("" ::"l"(o) : "memory");
        } else if (dm) {
          atomicAdd(&A.ctl[CTL_OUTSTANDING], delta);  // not waited for
        }
      }
      __syncwarp();  // orders the leader's atomics before the lanes' fence
      if (done) {
        active = false;
        ev = EV_NONE;
      }
      if (nfree > nin) {
        tick = __shfl_sync(kFull, tick, 0);
        const unsigned q = __popc(fm & lt_mask);
        if (((fm >> lane) & 1u) && q >= nin) ticket = (long long)(tick + (q - nin));
      }
      if (sm) base = __shfl_sync(kFull, base, 0);
      if (!FSL && nin) {
        const unsigned q = __popc(fm & lt_mask);
        const bool recv = ((fm >> lane) & 1u) && q < nin;
        Rec c = w.make_child(4u * w.pix);  // in splitting lanes: child 0's record, children differ in pix
        W::shfl_rec(c, recv ? nth_set_bit(sm, q / 3u) : lane);
        if (recv) {
          c.pix += q % 3u + 1u;
          w.load(c);
          active = true;
          fresh = START_CHILD;
        }
      }
      if (split) {
        w.on_split(A, acc);
        const unsigned i = __popc(sm & lt_mask);
        const SourceDev& S = A.src[w.src];
        const int cl = w.lvl() + 1;
        LC.add(A, S.inst, S.local, cl, 4u * w.pix, 4);
        // children 3 i + k - 1 >= nin to consecutive slots: the payloads, one
        // fence (which also waits for the warp's reductions in flight, so it
        // is paid once and not per record: 128^3 Stroemgren snapshot 0.268 ->
        // 0.252 ms, 24-grid batch 2.12 -> 1.99 ms), then the tags
        const unsigned j0 = 3u * i < nin ? (nin - 3u * i < 3u ? nin - 3u * i : 3u) : 0u;  // placed in this warp
        const unsigned long long slot0 = base + (3u * i + j0 - nin);
        Rec c = w.make_child(4u * w.pix);
        for (unsigned k = j0; k < 3u; ++k) {
          c.pix = 4u * w.pix + 1u + k;
          if (slot0 + (k - j0) < A.cap) W::template put<FSL>(&queue[slot0 + (k - j0)], c);
        }
        if (j0 < 3u) {
          __threadfence();
          const uint32_t tag = W::template tag_of<FSL>(c, sh_epoch);
          unsigned dropped = 0;
          for (unsigned k = j0; k < 3u; ++k) {
            if (slot0 + (k - j0) < A.cap) st_relaxed_u32(&queue[slot0 + (k - j0)].tag, tag);
            else ++dropped;
          }
          if (dropped) {
            set_status(A.ctl, RT_ERR_QUEUE_OVERFLOW);
            atomicAdd(&A.ctl[CTL_OUTSTANDING], (unsigned long long)(-(long long)dropped));
          }
        }
        w.become_child0();
        ev = EV_NONE;
        fresh = START_CHILD;
      }
    }
    // (2) turn tickets into packages
    uint32_t cell = 0;
    if (!active && ticket >= 0) {
      const unsigned long long tk = (unsigned long long)ticket;
      if (tk < A.n_roots) {
        const uint32_t ls = (uint32_t)(tk / A.npix0);
        const uint32_t p = (uint32_t)(tk - (unsigned long long)ls * A.npix0);
        w.load(W::root_rec((uint32_t)A.src_first + ls, (uint32_t)A.level0, p));
        fresh = START_ROOT;
      } else if (FSL && tk < qbase) {
        // a package halted by the previous trace continues from its cell
        const Rec q = *((const Rec*)A.res_in + (res_a + (tk - A.n_roots)));
        w.load(q);
        cell = W::cell_of_record(q);
        fresh = START_RESUMED;
      } else {
        const unsigned long long slot = tk - qbase;
        if (slot < A.cap) {
          Rec q;
          if (W::template poll<FSL>(&queue[slot], sh_epoch, q)) {
            w.load(q);
            fresh = START_CHILD;
          }
        }
      }
      if (fresh != NO_START) {
        ticket = -1;
        active = true;
      }
    }
    // (3) start the new packages, wherever they came from (one that starts
    //     outside the box is finished at the next (1))
    __syncwarp();
    if (fresh != NO_START) {
      const SourceDev& S = A.src[w.src];
      acc_switch(acc, w.nseg, S.inst, A, BB);
      if (FSL) w.set_rlim(A);
      if (fresh == START_ROOT) {
        if (FSL) acc.emitted += w.emit(S) * S.unit;
        else acc.emitted += S.unit;
        LC.add(A, S.inst, S.local, A.level0, w.pix, 1);
      }
      if (FSL && fresh == START_RESUMED) acc.resumed += (double)w.P * S.unit;
      if (!w.template start<FSL>(A, acc, FSL && fresh == START_RESUMED, cell)) {
        w.on_start_outside(A, acc);
        ev = EV_DONE;
      }
    }
    // (4) a warp with nothing to trace checks for the end of the trace
    const unsigned am = __ballot_sync(kFull, active);
    if (am == 0) {
      long long outst = 0;
      if (lane == 0) outst = (long long)ld_relaxed_u64(&A.ctl[CTL_OUTSTANDING]);
      outst = __shfl_sync(kFull, outst, 0);
      if (outst <= 0) break;
      const uint64_t now = global_ns();
      const unsigned backoff = idle.backoff;
      const bool moved = outst != idle.seen_out;
      const bool late = !moved && (long long)(now - idle.seen_ns) > A.timeout_ns;
      __syncwarp();
      if (late) {
        if (lane == 0) set_status(A.ctl, RT_ERR_TIMEOUT);
        break;
      }
      if (lane == 0) {
        if (moved) {
          idle.seen_out = outst;
          idle.seen_ns = now;
        }
        // (a longer sleep shows as latency where a trace has few packages,
        // up to a level of the ray tree each; 512 ns was no faster)
        idle.backoff = backoff < 1024 ? 2 * backoff : 1024;
      }
      __syncwarp();
      __nanosleep(backoff);
      continue;
    }
    if (lane == 0) {
      idle.backoff = 256;
      idle.seen_out = -1;  // the no-progress clock runs over one idle stretch only
    }
    // (5) trace a few segments
    if (active && ev == EV_NONE) {
      w.begin_visit();
      for (int it = 0; it < A.segs_per_iter; ++it) {
        ev = w.template step<FSL>(A, acc);
        if (ev != EV_NONE) break;
      }
    }
    // The lanes left the loop at different steps: reconverge them here, before
    // the warp-wide steps.  (Without this barrier the same kernel ran
    // 7-11 % slower on every workload measured.)
    __syncwarp();
    // (5b) the decisions that the segments left, for all lanes together: a
    //      lane's last segment (split, exit, halt, termination) runs here once
    //      per visit instead of inside the loop whenever one lane needs it
    //      (with the rates interleaved: 24 sources in an ionised 128^3 grid 9.67 ->
    //      7.62 ms, 1000 in a clumpy 256^3 grid 3.51 -> 2.71 ms)
    if constexpr (W::kStaged) {
      const bool left = ev == EV_RARE || ev == EV_TERM;
      if (__ballot_sync(kFull, left)) {
        float dep = 0.0f;
        const int at = w.idx;
        const bool first = left && w.r.hi == 0.0f;
        if (ev == EV_RARE) ev = w.template slow<FSL>(A, acc, dep);
        if (ev == EV_TERM) ev = w.template terminate<FSL>(A, acc, dep);
        __syncwarp();
        if (__ballot_sync(kFull, first)) w.deposit_first(first, at, dep);
        if (left && !first) w.deposit(at, dep);
      }
      if (active) ev = w.end_visit(A, acc, ev);
    }
    __syncwarp();
    // (6) halted packages go to the output store (one atomic per warp);
    //     from here on they are finished packages
    if (FSL) {
      const unsigned hm = __ballot_sync(kFull, ev == EV_HALT);
      if (hm) {
        const int leader = __ffs(hm) - 1;
        unsigned long long base = 0;
        if (lane == leader) base = atomicAdd(&A.ctl[CTL_HALTED], (unsigned long long)__popc(hm));
        base = __shfl_sync(kFull, base, leader);
        if (ev == EV_HALT) {
          const unsigned long long slot = base + __popc(hm & lt_mask);
          if (slot < A.halt_cap) w.store_halted((Rec*)A.halt_out + slot);
          else set_status(A.ctl, RT_ERR_QUEUE_OVERFLOW);
          ev = EV_DONE;
        }
      }
    }
  }
  acc.segments += w.nseg;
  // Where every lane of the block last worked on the same grid (or on none),
  // reduce the lanes' sums in shared memory first: 256 atomics onto one
  // word would serialise.
  __shared__ int sh_inst;
  if (threadIdx.x == 0) sh_inst = -1;
  __syncthreads();
  if (acc.inst >= 0) atomicMax(&sh_inst, acc.inst);
  __syncthreads();
  if (__syncthreads_and(acc.inst < 0 || acc.inst == sh_inst)) {
    for (int h = kBlock / 2; h > 0; h >>= 1) {
      if (threadIdx.x < h) {
        const LaneAcc& o = sh_acc[threadIdx.x + h];
        acc.emitted += o.emitted;
        acc.absorbed += o.absorbed;
        acc.escaped += o.escaped;
        acc.resumed += o.resumed;
        acc.halted += o.halted;
        acc.segments += o.segments;
        acc.fallbacks += o.fallbacks;
        acc.fallbacks_tau += o.fallbacks_tau;
      }
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      acc.inst = sh_inst;
      acc_flush(acc, A, BB);
    }
  } else {
    acc_flush(acc, A, BB);
  }
  // the block's reductions into its rows are complete and visible before
  // the rows are read back (from L2)
  __threadfence();
  __syncthreads();
  for (int i = threadIdx.x; i < A.blk_rows; i += blockDim.x) {
    const InstDev& I = A.inst[i];
    for (int k = 0; k < kAcc; ++k) {
      const double v = __ldcg(&brow[kBlkRow * i + k]);
      if (v != 0.0) atomicAdd(&I.acc[k], v);
    }
    const unsigned long long sg = __ldcg(reinterpret_cast<const unsigned long long*>(&brow[kBlkRow * i + kAcc]));
    if (sg) atomicAdd(&I.cnt[kCntSegments], sg);
    if (sh_bfb[2 * i]) atomicAdd(&I.cnt[kCntFallbacks], (unsigned long long)sh_bfb[2 * i]);
    if (sh_bfb[2 * i + 1]) atomicAdd(&I.cnt[kCntFallbacksTau], (unsigned long long)sh_bfb[2 * i + 1]);
  }
  for (int i = threadIdx.x; i < kShInst * kLevels; i += blockDim.x) {
    const int inst = i / kLevels, l = i - inst * kLevels;
    if (inst < A.ninst && sh_cnt[i]) {
      atomicAdd(&A.inst[inst].cnt[l], (unsigned long long)sh_cnt[i]);
      atomicAdd(&A.inst[inst].cnt[kLevels + l], sh_hsh[i]);
    }
  }
}

constexpr int kInitBlocks = 16;  // blocks of trace_init_kernel (they clear the queue at an epoch wrap)

// Resets the queue for pass `pass` of `passes`.  A trace may run as several
// passes over ranges of its sources; the status of earlier passes stays (the
// first error wins) and their queue use is folded into CTL_PEAK / CTL_PUSHED.
// Packages in flight (finite speed of light): at the first pass, mode
// FLIGHT_ADVANCE takes what the previous trace halted (at most in_cap
// records were stored) as this trace's input; every pass continues an equal
// share of them.
//
// Every pass takes the next epoch, and queue records carry its low 16 bits
// (QRec32).  Before an epoch whose low 16 bits would be 0 the launch clears
// the queue (all blocks, grid-stride) and takes the epoch after it: a record
// left in a slot that no trace has written for 2^16 - 1 epochs cannot then
// pass for a current one, and zeroed memory never does.  Every block reads
// the old epoch before it counts itself done in CTL_INIT_DONE; the block that
// counts last writes the control words (no block waits on another).
__global__ void trace_init_kernel(unsigned long long* ctl, uint4* queue, unsigned long long queue_u4,
                                  unsigned long long n_roots, int first_pass, int mode, unsigned long long in_cap,
                                  int pass, int passes) {
  __shared__ unsigned long long s_epoch;
  __shared__ int s_last;
  if (threadIdx.x == 0) s_epoch = *(volatile unsigned long long*)&ctl[CTL_EPOCH];
  __syncthreads();
  const unsigned long long old = s_epoch;
  const bool wrap = ((old + 1) & kEpochMask) == 0;
  if (wrap && queue) {
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < queue_u4;
         i += (unsigned long long)gridDim.x * blockDim.x)
      queue[i] = z;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(&ctl[CTL_INIT_DONE], 1ULL) == (unsigned long long)gridDim.x - 1ULL;
  }
  __syncthreads();
  if (threadIdx.x != 0 || !s_last) return;
  __threadfence();
  ctl[CTL_INIT_DONE] = 0;
  if (first_pass) {
    // a state rejected by an asynchronous upload stays reported until the
    // host has read it
    ctl[CTL_STATUS] = ctl[CTL_SET_ERR];
    ctl[CTL_PEAK] = 0;
    ctl[CTL_PUSHED] = 0;
    if (mode == FLIGHT_OFF) ctl[CTL_RESUME] = 0;
    else if (mode == FLIGHT_ADVANCE) ctl[CTL_RESUME] = ctl[CTL_HALTED] < in_cap ? ctl[CTL_HALTED] : in_cap;
    ctl[CTL_HALTED] = 0;
  } else {
    const unsigned long long t = ctl[CTL_TAIL];
    if (t > ctl[CTL_PEAK]) ctl[CTL_PEAK] = t;
    ctl[CTL_PUSHED] += t;
  }
  const unsigned long long nr = ctl[CTL_RESUME];
  const unsigned long long a = nr * (unsigned long long)pass / (unsigned long long)passes;
  const unsigned long long b = nr * (unsigned long long)(pass + 1) / (unsigned long long)passes;
  ctl[CTL_RES_A] = a;
  ctl[CTL_RES_B] = b;
  ctl[CTL_HEAD] = 0;
  ctl[CTL_TAIL] = 0;
  ctl[CTL_OUTSTANDING] = n_roots + (b - a);
  ctl[CTL_EPOCH] = old + (wrap ? 2ULL : 1ULL);
}

// Host-side launch helpers (called from api.cu).  `queue` / `queue_bytes`:
// the whole queue allocation (a multiple of 16 bytes), cleared when the epoch
// wraps.
cudaError_t launch_trace_init(unsigned long long* ctl, void* queue, size_t queue_bytes, unsigned long long n_roots,
                              int first_pass, int mode, unsigned long long in_cap, int pass, int passes,
                              cudaStream_t st) {
  if (queue_bytes % 16 != 0 || ((uintptr_t)queue & 15u) != 0) return cudaErrorInvalidValue;
  trace_init_kernel<<<kInitBlocks, 256, 0, st>>>(ctl, (uint4*)queue, queue_bytes / 16, n_roots, first_pass, mode,
                                                in_cap, pass, passes);
  return cudaGetLastError();
}

// Halting radii of the next trace from those of the previous one (finite
// speed of light): neu[0] = c_dt, neu[a] = old[a - 1] + c_dt, FP64, and
// their FP32 pairs.
__global__ void flight_table_kernel(const double* old, double* neu, float2* neu32, int n_new, double c_dt) {
  for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < n_new; a += gridDim.x * blockDim.x) {
    const double v = a == 0 ? c_dt : __dadd_rn(old[a - 1], c_dt);
    neu[a] = v;
    const float hi = __double2float_rn(v);
    neu32[a] = make_float2(hi, __double2float_rn(__dsub_rn(v, (double)hi)));
  }
}

cudaError_t launch_flight_table(const double* old, double* neu, float2* neu32, int n_new, double c_dt,
                                cudaStream_t st) {
  flight_table_kernel<<<(n_new + 255) / 256, 256, 0, st>>>(old, neu, neu32, n_new, c_dt);
  return cudaGetLastError();
}

constexpr int kMinBlocks64 = 2;
constexpr int kMinBlocks32 = TRACE_MIN_BLOCKS;

using TraceKernel = void (*)(TraceArgs);
template <bool FSL, bool FC>
static TraceKernel trace_instance32(int variant) {
  switch (variant) {
    case WALK_EXACT: return trace_kernel<Walk32<true, true, FC>, kMinBlocks32, FSL>;
    case WALK_ANY: return trace_kernel<Walk32<false, true, FC>, kMinBlocks32, FSL>;
    case WALK_ANY_PLAIN:
      if constexpr (!FSL) return trace_kernel<Walk32<false, false, FC>, kMinBlocks32, false>;
  }
  return nullptr;
}
// The instantiation for a launch; null for a combination that has none.
// fsl: finite speed of light (A.rlim*, res_in, halt_out set); fc: covering
// factor (A.fc; the FP64 walker tests that at run time).
static TraceKernel trace_instance(int precision, int fsl, int fc, int variant) {
  if (precision == RT_FP64)
    return fsl ? trace_kernel<Walk64, kMinBlocks64, true> : trace_kernel<Walk64, kMinBlocks64, false>;
  if (fsl) return fc ? trace_instance32<true, true>(variant) : trace_instance32<true, false>(variant);
  return fc ? trace_instance32<false, true>(variant) : trace_instance32<false, false>(variant);
}

cudaError_t trace_occupancy(int precision, int fsl, int fc, int variant, int block, int* blocks_per_sm) {
  const TraceKernel k = trace_instance(precision, fsl, fc, variant);
  if (!k || block != kBlock) return cudaErrorInvalidValue;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, block, 0);
}

cudaError_t launch_trace(int precision, int fsl, int variant, const TraceArgs& A, int grid, int block,
                         cudaStream_t st) {
  const TraceKernel k = trace_instance(precision, fsl, A.fc, variant);
  if (!k || block != kBlock) return cudaErrorInvalidValue;
  k<<<grid, block, 0, st>>>(A);
  return cudaGetLastError();
}

// Direction table: for each pixel of levels 0..L (level l starts at entry
// 4 (4^l - 1)), two float4: (hi.x, hi.y, hi.z, diag) and (lo.x, lo.y, lo.z, 0)
// with hi + lo the FP64 direction of pix2vec64.
__global__ void direction_table_kernel(int level, float4* tab) {
  const unsigned long long npix = 12ULL << (2 * level);
  const size_t base = (size_t)4 * (((size_t)1 << (2 * level)) - 1);
  for (unsigned long long p = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; p < npix;
       p += (unsigned long long)gridDim.x * blockDim.x) {
    double v[3];
    const int diag = pix2vec64(level, (uint32_t)p, v);
    float hi[3], lo[3];
    for (int i = 0; i < 3; ++i) {
      hi[i] = (float)v[i];
      lo[i] = (float)(v[i] - (double)hi[i]);
    }
    tab[2 * (base + p)] = make_float4(hi[0], hi[1], hi[2], diag ? 1.0f : 0.0f);
    tab[2 * (base + p) + 1] = make_float4(lo[0], lo[1], lo[2], 0.0f);
  }
}

cudaError_t launch_direction_table(int level, float4* tab, cudaStream_t st) {
  direction_table_kernel<<<152 * 8, 256, 0, st>>>(level, tab);
  return cudaGetLastError();
}

// Self-check of the FP32 direction bound: max over the pixels of `level` of
// max_i |n32_i - n64_i|, written to out[0] (as the bit pattern of a positive
// double, so atomicMax on the integer view orders it correctly).
__global__ void direction_error_kernel(int level, unsigned long long* out) {
  const unsigned long long npix = 12ULL << (2 * level);
  double worst = 0.0;
  for (unsigned long long p = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; p < npix;
       p += (unsigned long long)gridDim.x * blockDim.x) {
    double n64[3];
    float n32[3];
    pix2vec64(level, (uint32_t)p, n64);
    pix2vec32(level, (uint32_t)p, n32);
    for (int i = 0; i < 3; ++i) worst = fmax(worst, fabs((double)n32[i] - n64[i]));
  }
  atomicMax(out, (unsigned long long)__double_as_longlong(worst));
}

cudaError_t launch_direction_check(int level, unsigned long long* out, cudaStream_t st) {
  direction_error_kernel<<<152 * 8, 256, 0, st>>>(level, out);
  return cudaGetLastError();
}

}  // namespace rtg
