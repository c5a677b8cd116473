// Resident evaluations: states small enough that every CTA of one launch holds its own tile.
//
// A launch runs a sequence of evaluations of H(t) (Runge-Kutta stages, the start of the
// derivative history, predictor-corrector steps; Sec. I.B) without leaving the GPU.  The state is
// cut into contiguous tiles of 2^t indices, one per CTA (several, when a caller limits the CTAs or
// the tiles outnumber them).  A thread owns the same amplitudes through the launch: y, the
// derivatives and the Runge-Kutta accumulator are read and written by that thread alone, in
// registers while a thread owns at most two 16-byte slots, else in global memory (they stay in
// L2).  Only the vector that H acts on next (the predictor, a stage input, or y) is seen by
// other threads: the CTA's own tile of it stays in shared memory, and a copy goes to one of two
// exchange vectors in global memory, from where the CTAs whose products flip bits above t fetch
// it as whole tiles.
//
// Exchange: products are sorted by the bits they flip above t ("partner" tiles; all products of
// one partner share one copy).  When a tile is done the CTA raises the tile's flag; one warp per
// CTA waits for its partners' flags, one by one, and starts a bulk copy (cp.async.bulk, completion
// on an mbarrier) of each partner tile as soon as it is up, while the other warps work on the
// products inside the tile.  The partner relation is symmetric, so having a partner's data also
// says that it no longer reads the exchange vector written next; no CTA waits for all others.
//
// Another warp does the scalar FP64 work beside them (coefficients of the next evaluation, the sum
// of the last one's error partials): on this GPU an FP64 instruction of a warp holds its
// multiprocessor's pipe for about 19 cycles, so reducing by shuffles in every warp would take
// longer than a small state's step.
//
// Up to 16 tiles run as one thread-block cluster and push their tiles into one another's shared
// memory instead: no flags, no trip through L2.  A push reports its completion at its destination
// only, so a CTA cannot tell when its own tile has been read; it keeps two (cluster_set): the tile of
// evaluation e + 1 is written beside that of e and over that of e - 1.  That one is free by then: a
// partner sends its tile of e only when it has finished e - 1, for which it needed all of this CTA's
// tile of e - 1, and no thread writes before it has seen every partner's tile of e.
//
// Measured, microseconds per predictor-corrector step (before: one launch per layout pass, replayed
// from a graph, each on as many CTAs as the state has 64 KiB tiles):
//   complex64, nonlinear path: n = 8 11 -> 1.8, n = 12 31 -> 2.4, n = 16 43 -> 4.2, n = 18 46 -> 8.5, n = 20 50 -> 35
//   complex128, linear path:   n = 10 20 -> 3.6, n = 14 68 -> 4.9, n = 16 71 -> 11, n = 18 72 -> 42
// An exchange takes about 0.8 us in a cluster and 1.5 us through memory (from the last store to the
// first partner read); the rest of a small state's step is dependent shared-memory reads and, in
// complex128, FP64 latency.  Counters: n = 12 complex64 waits (issue slots 25% busy on 16 multiprocessors,
// barriers the first stall); n = 20 keeps shared memory's pipe 46% busy with the partners' reads (16
// bytes per product and slot) and issue slots 42%, the rest is barriers between its phases, with one CTA
// per multiprocessor; complex128 n = 16 keeps the FP64 pipe 81% busy.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "aqc_internal.h"
#include "kernel_shape.h"

namespace aqc {

namespace {

template <typename R>
struct RT;
template <>
struct RT<float> {
  using C2 = float2;
  static constexpr int H = 2;  // amplitudes per 16-byte slot
};
template <>
struct RT<double> {
  using C2 = double2;
  static constexpr int H = 1;
};

template <typename R>
struct RPlain {  // X string with a real coefficient: place of the partner, coefficient
  uint32_t off;
  R c;
};
struct RBase {  // the same before the group weight
  double coef;
  uint32_t off;
  int group;
};
template <typename R>
struct RGen {  // hop or general product: mask, phases, place, effective coefficients
  uint32_t x, zm, zm2, off;
  R cr, ci, cr2, ci2;
};
template <typename R>
struct RScal {        // diagonal of one evaluation
  R dt[256];          // identity prefactors plus the byte-table class's energy, by clause count
  R cw[kMaxClasses];  // weights of the other clause classes
};

constexpr uint32_t kResPolls = 1u << 22;  // flag and mbarrier polls before a wait gives up
constexpr int kService = 128;             // threads beside those that own amplitudes: four warps

// threads that own amplitudes, at most: sixteen slots per thread need more registers than 512 threads
// (and the service warps) leave
__host__ __device__ constexpr int owners(int slots) { return slots >= 8 ? kResMaxThreads / 2 : kResMaxThreads; }

__host__ __device__ inline size_t up16(size_t v) { return (v + 15) & ~(size_t)15; }

// shared memory: [own tile][nbuf partner tiles][clause bytes][weights][bases][plain x2][general x2]
// [Z x2][Z masks][scalars x2][reductions x2][lane sums][mbarriers]
template <typename R>
struct ResSmem {
  size_t code, w, base, pl, gen, z, zm, scal, red, lane, bar, total;
  __host__ __device__ ResSmem(uint32_t tsize, int nbuf, int np, int ng, int nz, int nth, bool dred) {
    code = up16((size_t)tsize * (1 + nbuf) * 2 * sizeof(R));
    w = up16(code + tsize);
    base = up16(w + 3 * kResMaxEvals * sizeof(double));
    pl = up16(base + (size_t)np * sizeof(RBase));
    gen = up16(pl + 2 * (size_t)np * sizeof(RPlain<R>));
    z = up16(gen + 2 * (size_t)ng * sizeof(RGen<R>));
    zm = up16(z + 2 * (size_t)nz * sizeof(R));
    scal = up16(zm + (size_t)nz * sizeof(uint32_t));
    red = up16(scal + 2 * sizeof(RScal<R>));
    lane = up16(red + 2 * (size_t)nth * (dred ? sizeof(double) : sizeof(R)));
    bar = lane + 8 * (kResMaxEvals + 1) * sizeof(double);
    total = bar + 2 * (size_t)(nbuf > 0 ? nbuf : 1) * sizeof(uint64_t);
  }
};

__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }

__device__ __forceinline__ unsigned flag_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void flag_release(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint32_t b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(b), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(b) : "memory");
}
__device__ __forceinline__ bool bar_try(uint32_t b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(b), "r"(parity)
      : "memory");
  return ok != 0u;
}
// bounded wait; ends early when another warp of the CTA has given up
__device__ __forceinline__ bool bar_wait(uint32_t b, uint32_t parity, const volatile int* abort) {
  for (uint32_t i = 0; i < kResPolls; i++) {
    if (bar_try(b, parity)) return true;
    if (*abort) return false;
  }
  return false;
}
__device__ __forceinline__ void expect(uint32_t b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(b), "r"(bytes) : "memory");
}
// the wait at the end of a launch that gave up: both phases of a barrier, short
__device__ __forceinline__ bool bar_wait_short(uint32_t b, uint32_t parity) {
  for (uint32_t i = 0; i < (1u << 14); i++)
    if (bar_try(b, parity)) return true;
  return false;
}
// bytes from global memory into shared memory (both 16-byte aligned), counted on b
__device__ __forceinline__ void tile_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t b) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst), "l"(src),
      "r"(bytes), "r"(b)
      : "memory");
}
// bytes from this CTA's shared memory into that of CTA `rank` of the cluster at the same place, counted
// on its barrier
__device__ __forceinline__ void tile_push(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t b, uint32_t rank) {
  asm volatile(
      "{\n .reg .b32 d, m;\n mapa.shared::cluster.u32 d, %0, %4;\n mapa.shared::cluster.u32 m, %3, %4;\n"
      " cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [d], [%1], %2, [m];\n}\n" ::"r"(dst),
      "r"(src), "r"(bytes), "r"(b), "r"(rank)
      : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive;\nbarrier.cluster.wait;\n" ::: "memory");
}
__device__ __forceinline__ void proxy_fence_shared() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async;\n" ::: "memory"); }

template <typename C2, int H>
__device__ __forceinline__ void unpack(const float4& x, C2 (&v)[H]) {
  const C2* xs = reinterpret_cast<const C2*>(&x);
#pragma unroll
  for (int q = 0; q < H; q++) v[q] = xs[q];
}
template <typename C2, int H>
__device__ __forceinline__ float4 pack(const C2 (&v)[H]) {
  float4 x;
  C2* xs = reinterpret_cast<C2*>(&x);
#pragma unroll
  for (int q = 0; q < H; q++) xs[q] = v[q];
  return x;
}

// hi + lo + inc as an exact two-sum renormalised into (hi, lo): the compensated corrector
__device__ __forceinline__ float add_compensated(float hi, float& lo, float inc) {
  const float s = __fadd_rn(hi, inc);
  const float bp = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(inc, bp));
  const float l = __fadd_rn(lo, e);
  const float h = __fadd_rn(s, l);
  lo = __fsub_rn(l, __fsub_rn(h, s));
  return h;
}
__device__ __forceinline__ double add_compensated(double hi, double&, double inc) { return hi + inc; }

// warp sum of v in lane order; the total in lane 0
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Kind of evaluation e of the launch: 1..4 Runge-Kutta stage, 5 start of the derivative history,
// 0 predictor-corrector step; 6 H psi, 7 <psi|H|psi>.
__device__ __forceinline__ int kind_of(const ResParams& P, int e) {
  if (P.single) return P.single;
  if (e < 4 * P.n_rk) return 1 + (e & 3);
  return (P.hist && e == 4 * P.n_rk) ? 5 : 0;
}

// Coefficients of the off-diagonal products at weights w (one warp).
template <typename R>
__device__ __forceinline__ void coefficients(const ResParams& P, const double* w, const RBase* base, RPlain<R>* pl,
                                             RGen<R>* gen) {
  const DevTables* tab = P.tab;
  const double w0 = w[0], w1 = w[1], w2 = w[2];
  auto pick = [&](int g) { return g == 0 ? w0 : (g == 1 ? w1 : w2); };
  const int lane = threadIdx.x & 31;
  for (int k = lane; k < P.np; k += 32) {
    const RBase d = base[k];
    pl[k] = RPlain<R>{d.off, (R)(d.coef * pick(d.group))};
  }
  for (int k = lane; k < P.ng; k += 32) {
    const DevFlip d = tab->flips[P.rt->idx[P.np + k]];
    double v[4] = {0.0, 0.0, 0.0, 0.0};  // c i^ipow of the product and of its companion
    auto phased = [](double c, int ipow, double* o) {
      o[0] = (ipow & 1) ? 0.0 : ((ipow & 2) ? -c : c);
      o[1] = (ipow & 1) ? ((ipow & 2) ? -c : c) : 0.0;
    };
    phased(d.coef * pick(d.group), d.ipow, v);
    if (d.has2) phased(d.coef2 * pick(d.group2), d.ipow2, v + 2);
    gen[k] = RGen<R>{d.x, d.zm, d.has2 ? d.zm2 : 0u, gen[k].off, (R)v[0], (R)v[1], (R)v[2], (R)v[3]};
  }
}

// Coefficients of the diagonal at weights w (one warp).
template <typename R>
__device__ __forceinline__ void diagonal_of(const ResParams& P, const double* w, R* zc, RScal<R>* sc,
                                            const double (&ident)[3], int nz, int ncls, double tscale, int tgroup) {
  const DevTables* tab = P.tab;
  const double w0 = w[0], w1 = w[1], w2 = w[2];
  auto pick = [&](int g) { return g == 0 ? w0 : (g == 1 ? w1 : w2); };
  const int lane = threadIdx.x & 31;
  for (int k = lane; k < nz; k += 32) zc[k] = (R)(tab->z[k].coef * pick(tab->z[k].group));
  const R dconst = (R)(ident[0] * w0 + ident[1] * w1 + ident[2] * w2);
  if (P.dcode) {
    const R wt = (R)(tscale * pick(tgroup));
    for (int k = lane; k <= P.ncode; k += 32) sc->dt[k] = fma_(wt, (R)k, dconst);
    if (ncls > 1)
      for (int k = lane; k < ncls; k += 32) sc->cw[k] = (R)(tab->classes[k].scale * pick(tab->classes[k].group));
  } else {
    if (lane == 0) sc->dt[0] = dconst;
    for (int k = lane; k < ncls; k += 32) sc->cw[k] = (R)(tab->classes[k].scale * pick(tab->classes[k].group));
  }
}

__device__ __forceinline__ int count_clauses(const DevTables* __restrict__ tab, int pen, int b, int e, uint32_t z) {
  int cnt = 0;
  for (int k = b; k < e; k++) {
    const int o = 1 - __popc(tab->clause_mask[k] & z);
    cnt += pen == 0 ? (o != 0) : o * o;
  }
  return cnt;
}

// -v where bit 0 of `odd` is set
__device__ __forceinline__ float negate_if(float v, uint32_t odd) { return __uint_as_float(__float_as_uint(v) ^ (odd << 31)); }
__device__ __forceinline__ double negate_if(double v, uint32_t odd) {
  return __hiloint2double((int)((uint32_t)__double2hiint(v) ^ (odd << 31)), __double2loint(v));
}
// Diagonal parts beside the table lookup, for the consecutive indices of a slot: other clause classes and
// Z strings, each taken once for both.  (One amplitude at a time, masks read from memory, 120 strings made a step
// at n = 20 take 265 us; two layout passes took 100.)
template <typename R>
struct RSlot {
  R d[RT<R>::H];
};
template <typename R>
__device__ __noinline__ RSlot<R> other_diagonal(const DevTables* tab, const RScal<R>& sc, const R* zc, const uint32_t* zm,
                                                int tcls, int code0, int code1, uint32_t z) {
  constexpr int H = RT<R>::H;
  RSlot<R> r;
#pragma unroll
  for (int q = 0; q < H; q++) r.d[q] = (R)0;
  for (int cc = 0; cc < tab->n_classes; cc++) {
    if (cc == tcls) continue;
    const DevClass cl = tab->classes[cc];
    const bool derived = cl.derived && tcls >= 0;
    const int b = derived ? cl.dbegin : cl.begin, e = derived ? cl.dend : cl.end;
#pragma unroll
    for (int q = 0; q < H; q++) {
      const int cnt = count_clauses(tab, cl.pen, b, e, z + (uint32_t)q);
      r.d[q] = fma_(sc.cw[cc], (R)(derived ? (q ? code1 : code0) - cnt : cnt), r.d[q]);
    }
  }
  const int nz = tab->n_z;
#pragma unroll 4
  for (int m = 0; m < nz; m++) {
    const uint32_t x = zm[m];
    const R c = negate_if(zc[m], (uint32_t)__popc(x & z));
    r.d[0] += c;
    if (H == 2) r.d[H - 1] += negate_if(c, x);
  }
  return r;
}

// All threads of the CTA, from the loop of any role.
__device__ __forceinline__ void cta_sync() { asm volatile("bar.sync 0;\n" ::: "memory"); }

// S slots per thread: a tile is S x (threads that own amplitudes) slots.  REG: the owned vectors
// stay in registers for the launch and the CTA has one tile; otherwise a CTA walks its tiles and
// the owned vectors come from global memory, a quarter tile at a time through the partner buffers
// (S >= 4) or one slot ahead.  Per amplitude all variants run the same operations in the same
// order.  PEC: predictor-corrector steps; otherwise the start-up and single evaluations.
//
// The warps take roles, each with its own loop over the evaluations: owners, the coefficients of
// the next evaluation's products, those of its diagonal, the sums of the last one's error
// partials, and the tile copies.
// The body runs as one tile (number `cta` of G tiles or CTAs) of the state that P describes; inst: the
// batch member, whose results go to its record (null: to P.slots).
//
// CLU: the CTAs are one thread-block cluster (at most 16, one slot per thread).  A finished tile goes
// straight into the partners' shared memory (cp.async.bulk between CTAs, completion on the
// partner's mbarrier), into one of two sets of tiles (the own one, then the partners') by the
// evaluation's parity: having a partner's data of one evaluation says that it is past the reads of
// the set written next, and that it has all of what this CTA pushed before.
template <typename R, int S, bool REG, bool PEC, bool COMP, bool CLU>
__device__ __forceinline__ void resident_body(const ResParams& P, const uint32_t cta, const uint32_t G,
                                              BatchInst* const inst) {
  using C2 = typename RT<R>::C2;
  constexpr int H = RT<R>::H;
  constexpr int A = S * H;  // amplitudes per thread and tile
  constexpr bool kComp = COMP && sizeof(R) == 4;
  constexpr bool kStream = PEC && !REG && !kComp && S >= 4;
  constexpr int SC = S / 4 > 0 ? S / 4 : 1;  // slots per streamed quarter tile
  using RED = typename std::conditional<REG, R, double>::type;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ ResStatic sh;
  ResPartner* const s_part = sh.part;
  ResRun* const s_run = sh.run;
  volatile int& s_abort = sh.abort;
  double* const s_err = sh.err;

  const DevTables* tab = P.tab;
  const int nth = (int)blockDim.x - kService, nwarps = nth >> 5;
  const int tid = threadIdx.x, lane = tid & 31;
  const bool owner = tid < nth;
  const int svc = (tid - nth) >> 5;  // service warp 0..3
  const uint32_t tsize = 1u << P.t, tmask = tsize - 1u, tbytes = tsize * (uint32_t)sizeof(C2);
  const uint32_t ntiles = 1u << (P.n - P.t);
  const int np = P.np, ng = P.ng, nz = tab->n_z, ncls = tab->n_classes;
  const int nd = P.npart, nbuf = P.nbuf;  // partner tiles (beside the own one) and their buffers
  const int nq = nd + (kStream && nbuf > 0 ? 4 : 0);  // ring entries per tile visit
  const bool ring = nbuf > 0 && (S >= 4 || nd > nbuf);  // else every partner has a buffer of its own
  const int tcls = P.dcode ? tab->table_class : -1;
  const int E = P.evals;
  const bool multi = ntiles > G;  // several tiles per CTA
  const ResSmem<R> M(tsize, nbuf, np, ng, nz, nth, !REG);
  C2* const xs = reinterpret_cast<C2*>(smem);
  uint8_t* const s_code = smem + M.code;
  double* const s_w = reinterpret_cast<double*>(smem + M.w);
  RBase* const s_base = reinterpret_cast<RBase*>(smem + M.base);
  RPlain<R>* const s_pl = reinterpret_cast<RPlain<R>*>(smem + M.pl);
  RGen<R>* const s_gen = reinterpret_cast<RGen<R>*>(smem + M.gen);
  R* const s_z = reinterpret_cast<R*>(smem + M.z);
  uint32_t* const s_zm = reinterpret_cast<uint32_t*>(smem + M.zm);
  RScal<R>* const s_sc = reinterpret_cast<RScal<R>*>(smem + M.scal);
  RED* const s_red = reinterpret_cast<RED*>(smem + M.red);           // [parity][nth]
  double* const s_lane = reinterpret_cast<double*>(smem + M.lane);  // [E + 1][8]
  const uint32_t full0 = saddr(smem + M.bar), empty0 = full0 + 8u * (uint32_t)nbuf;

  if (tid == 0) {
    s_abort = 0;
    for (int b = 0; b < nbuf; b++) {
      bar_init(full0 + 8u * b, 1);
      bar_init(empty0 + 8u * b, (uint32_t)nwarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  for (int k = tid; k <= nd; k += blockDim.x) s_part[k] = P.rt->part[k];
  for (int k = tid; k < P.nruns; k += blockDim.x) s_run[k] = P.rt->run[k];
  for (int k = tid; k < nz; k += blockDim.x) s_zm[k] = tab->z[k].zm;
  for (int k = tid; k < 3 * E; k += blockDim.x)
    s_w[k] = P.wdev ? P.wdev[(size_t)P.wstride * (k / 3) + k % 3] : P.w[k];
  __syncthreads();
  // a product's place in shared memory: its flip inside the tile, and its partner's buffer when
  // every partner has one (XOR with a slot's byte offset)
  auto place = [&](uint32_t x) {
    uint32_t p = 0;
    if (!ring)
      while (s_part[p].hi != (x >> P.t)) p++;
    return (x & tmask) * (uint32_t)sizeof(C2) | p * tbytes;
  };
  for (int k = tid; k < np; k += blockDim.x) {
    const DevFlip d = tab->flips[P.rt->idx[k]];
    s_base[k] = RBase{d.coef, place(d.x), d.group};
  }
  for (int k = tid; k < ng; k += blockDim.x) s_gen[k].off = s_gen[ng + k].off = place(tab->flips[P.rt->idx[np + k]].x);
  __syncthreads();
  if (CLU) cluster_sync();  // every CTA's barriers are ready for the others' copies

  // copies of partner tiles (and of owned quarter tiles) for one visit of a tile; q0: ring entries
  // so far, visit: tile visits so far
  auto copy_in = [&](uint32_t tile, const C2* xin, int e, int latest, uint32_t q0) {
    auto give_up = [&]() {
      s_abort = 1;
      P.slots[kSlotFault] = 1.0;
    };
    auto ready = [&](uint32_t other) {  // the partner has published this evaluation's source
      if (e == 0) return true;
      uint32_t polls = 0;
      while (flag_acquire(P.flags + kResFlagStride * other) < (unsigned)e) {
        if (++polls > kResPolls || s_abort) return false;
        if (polls > 256u) __nanosleep(64);
      }
      return true;
    };
    if (!ring) {
      if (lane == 0) expect(full0, (uint32_t)nd * tbytes);
      __syncwarp();
      for (int p = lane; p < nd; p += 32) {
        const uint32_t other = tile ^ s_part[p + 1].hi;
        if (!ready(other)) {
          give_up();
          break;
        }
        proxy_fence();  // the partner's stores, seen by its flag, before the asynchronous copy
        tile_copy(saddr(xs + (size_t)(1 + p) * tsize), xin + ((size_t)other << P.t), tbytes, full0);
      }
    } else if (lane == 0) {
      uint32_t b = q0 % (uint32_t)nbuf, use = q0 / (uint32_t)nbuf;
      for (int p = 0; p < nq; p++) {
        const uint32_t other = p < nd ? tile ^ s_part[p + 1].hi : tile;
        if ((use > 0 && !bar_wait(empty0 + 8u * b, (use - 1u) & 1u, &s_abort)) || (p < nd && !ready(other))) {
          give_up();
          break;
        }
        proxy_fence();
        const uint32_t dst = saddr(xs + (size_t)(1u + b) * tsize), bb = full0 + 8u * b;
        expect(bb, tbytes);
        if (p < nd) {
          tile_copy(dst, xin + ((size_t)other << P.t), tbytes, bb);
        } else {
          const uint32_t part = tbytes / 4;
          const size_t z = ((size_t)tile << P.t) + (size_t)(p - nd) * (tsize / 4);
          const void* v[4] = {P.y, P.f[latest & 3], P.f[(latest - 1) & 3], P.f[(latest - 2) & 3]};
#pragma unroll
          for (int i = 0; i < 4; i++) tile_copy(dst + i * part, reinterpret_cast<const C2*>(v[i]) + z, part, bb);
        }
        if (++b == (uint32_t)nbuf) {
          b = 0;
          use++;
        }
      }
    }
    __syncwarp();
  };
  auto copies_land = [&]() {  // at the end of a launch that gave up (one warp): the copies under way, bounded
    const int used = CLU ? 2 : (ring ? nbuf : (nbuf > 0 ? 1 : 0));
    for (int b = lane; b < used; b += 32)
      for (uint32_t par = 0; par < 2; par++) (void)bar_wait_short(full0 + 8u * b, par);
    __syncwarp();
  };
  auto all_sync = [&]() { asm volatile("bar.sync 2, %0;\n" ::"r"((int)blockDim.x) : "memory"); };
  const C2* const src0 = reinterpret_cast<const C2*>(P.src);
  C2* const XA = reinterpret_cast<C2*>(P.xout[0]);
  C2* const XO = reinterpret_cast<C2*>(P.xout[1]);
  // a[] holds f_latest; at a start-up f_k is known for k < step0, later for k <= step0
  const int first_latest = P.single ? 0 : (P.n_rk > 0 || P.hist ? P.step0 - 1 : P.step0);
  int latest = first_latest;
  uint32_t q0 = 0, visit = 0;

  if (owner) {
    C2* const Y = reinterpret_cast<C2*>(P.y);
    C2* const YO = reinterpret_cast<C2*>(P.yout);
    C2* const ACC = reinterpret_cast<C2*>(P.acc);
    C2* const YL = reinterpret_cast<C2*>(P.ylo);
    auto F = [&](int k) { return reinterpret_cast<C2*>(P.f[k & 3]); };  // f_k's ring slot
    const R h = (R)P.h;
    const double e24 = P.h / 24.0;
    const R h24 = (R)e24, h24lo = sizeof(R) == 8 ? (R)0 : (R)(e24 - (double)h24);
    const R c9 = (R)9 * h24, c19 = (R)19 * h24, c5 = (R)5 * h24;
    const R c64 = (R)64 * h24, p55 = (R)55 * h24, p59 = (R)59 * h24, p37 = (R)37 * h24, p9 = (R)9 * h24;
    const bool others = nz > 0 || ncls > (tcls >= 0 ? 1 : 0);
    // y, f of the last three steps, Runge-Kutta accumulator and low part of y of one slot
    struct Owned {
      C2 y[H], a[H], b[H], c[H], rk[H], yl[H];
    };
    // The past's part of the corrector (cq) and of the predictor (pq): in FP64 with y in both, so that
    // one multiply-add with f_{n+1} completes either (9 and 9 + 55 = 64 times h/24); in FP32 the
    // weighted sums of derivatives, before the scaling by h/24.
    auto past = [&](const Owned& w, int q, int kind, C2& cq, C2& pq) {
      const C2 &y = w.y[q], &a = w.a[q], &b = w.b[q], &c = w.c[q];
      if (sizeof(R) == 8) {
        cq = kind == 0 ? C2{fma_(c19, a.x, fma_(-c5, b.x, fma_(h24, c.x, y.x))),
                            fma_(c19, a.y, fma_(-c5, b.y, fma_(h24, c.y, y.y)))}
                       : y;  // (the start of the history corrects nothing)
        pq = C2{fma_(-p59, a.x, fma_(p37, b.x, fma_(-p9, c.x, cq.x))),
                fma_(-p59, a.y, fma_(p37, b.y, fma_(-p9, c.y, cq.y)))};
      } else {
        cq = C2{fma_((R)19, a.x, fma_((R)-5, b.x, c.x)), fma_((R)19, a.y, fma_((R)-5, b.y, c.y))};
        pq = C2{fma_((R)-59, a.x, fma_((R)37, b.x, (R)-9 * c.x)), fma_((R)-59, a.y, fma_((R)37, b.y, (R)-9 * c.y))};
      }
    };
    auto load = [&](const C2* v, C2 (&d)[H]) { unpack<C2, H>(*reinterpret_cast<const float4*>(v), d); };
    auto store = [&](C2* v, const C2 (&d)[H]) { *reinterpret_cast<float4*>(v) = pack<C2, H>(d); };
    const int j0 = tid * H, js = nth * H;  // tile position of the first slot, slot stride
    const bool act = j0 < (int)tsize;      // tiles below one slot per thread: some idle
    const uint32_t jb = (uint32_t)j0 * sizeof(C2), jsb = (uint32_t)js * sizeof(C2);
    const int jsl = 31 - __clz(js);
    Owned o[REG ? S : 1];
    if (REG && act && !P.single) {
#pragma unroll
      for (int s = 0; s < S; s++) {
        const uint32_t z = (cta << P.t) + (uint32_t)(j0 + s * js);
        load(Y + z, o[s].y);
        if (latest >= 0) load(F(latest) + z, o[s].a);
        if (latest >= 1) load(F(latest - 1) + z, o[s].b);
        if (latest >= 2) load(F(latest - 2) + z, o[s].c);
        if (kComp) load(YL + z, o[s].yl);
      }
    }
    const C2* xin = src0;
    C2* xout = XA;
    RED final0 = (RED)0;  // the last evaluation's first reduction (||y||^2, Re <src|H|src>)
    for (int e = 0; e < E; e++) {
      const int kind = PEC ? 0 : kind_of(P, e), par = e & 1;
      const bool last = e == E - 1;
      const RPlain<R>* const pl = s_pl + par * np;
      const RGen<R>* const gen = s_gen + par * ng;
      const RScal<R>& sc = s_sc[par];
      RED red0 = (RED)0, red1 = (RED)0;
      // the set of tiles that this evaluation reads, and where the own tile of the next one goes
      const uint32_t set = CLU ? (uint32_t)cluster_set(e) * (1u + (uint32_t)nd) : 0u;
      const unsigned char* const tiles = smem + (size_t)set * tbytes;
      C2* const xs_e = xs + (size_t)set * tsize;
      C2* const xs_next = CLU ? xs + (size_t)((uint32_t)cluster_set(e + 1) * (1u + (uint32_t)nd)) * tsize : xs;
      for (uint32_t tile = cta; tile < ntiles; tile += G, visit++) {
        const uint32_t zb = tile << P.t;
        if (e == 0 || multi) {  // the own tile and its clause bytes (then kept up to date in place)
          if (multi) cta_sync();  // readers of the previous tile are done
          if (REG) {
            for (uint32_t j = j0; j < tsize; j += js)
              *reinterpret_cast<float4*>(xs + j) = __ldcg(reinterpret_cast<const float4*>(xin + zb + j));
            if (tcls >= 0)
              for (uint32_t j = j0; j < tsize; j += js)
#pragma unroll
                for (int q = 0; q < H; q++) s_code[j + q] = P.dcode[zb + j + q];
          } else if (act) {  // on every visit: all loads at once
            float4 v[REG ? 1 : S];
#pragma unroll
            for (int s = 0; s < S; s++) v[REG ? 0 : s] = __ldcg(reinterpret_cast<const float4*>(xin + zb + (uint32_t)(j0 + s * js)));
            if (tcls >= 0) {
              if (tsize >= 16u) {
                for (uint32_t j = 16u * tid; j < tsize; j += 16u * nth)
                  *reinterpret_cast<float4*>(s_code + j) = __ldg(reinterpret_cast<const float4*>(P.dcode + zb + j));
              } else {
#pragma unroll
                for (int q = 0; q < H; q++) s_code[j0 + q] = P.dcode[zb + (uint32_t)j0 + q];
              }
            }
#pragma unroll
            for (int s = 0; s < S; s++) *reinterpret_cast<float4*>(xs + (j0 + s * js)) = v[REG ? 0 : s];
          }
          cta_sync();
        }
        R ar[A], ai[A];
#pragma unroll
        for (int g = 0; g < A; g++) ar[g] = ai[g] = (R)0;
        // X strings with real coefficients [k, end) out of the tiles from `t` on, one 16-byte load per
        // slot (two 8-byte loads, which need no swap for a flip of index bit 0, hit each bank twice)
        auto plain = [&](const unsigned char* t, int k, int end) {
          constexpr int U = S >= 4 ? 1 : 4 / S;  // products in flight
          auto some = [&](auto count, int k) {
            constexpr int C = decltype(count)::value;
            RPlain<R> f[C];
            float4 v[C][S];
#pragma unroll
            for (int i = 0; i < C; i++) {
              f[i] = pl[k + i];
              const uint32_t at = jb ^ (f[i].off & ~15u);
#pragma unroll
              for (int s = 0; s < S; s++) v[i][s] = *reinterpret_cast<const float4*>(t + (at ^ ((uint32_t)s * jsb)));
            }
#pragma unroll
            for (int i = 0; i < C; i++) {
              const bool sw = H == 2 && (f[i].off & 15u);
#pragma unroll
              for (int s = 0; s < S; s++) {
                C2 u[H];
                unpack<C2, H>(v[i][s], u);
#pragma unroll
                for (int q = 0; q < H; q++) {
                  const C2 x = sw ? u[H - 1 - q] : u[q];
                  ar[s * H + q] = fma_(f[i].c, x.x, ar[s * H + q]);
                  ai[s * H + q] = fma_(f[i].c, x.y, ai[s * H + q]);
                }
              }
            }
          };
          if constexpr (S >= 4) {  // one product at a time, up to eight slots' loads at once
#pragma unroll 1
            for (; k < end; k++) {
              const RPlain<R> f = pl[k];
              const uint32_t at = jb ^ (f.off & ~15u);
              const bool sw = H == 2 && (f.off & 15u);
              constexpr int L = S < 8 ? S : 8;  // loads in flight
#pragma unroll
              for (int s0 = 0; s0 < S; s0 += L) {
                float4 v[L];
#pragma unroll
                for (int i = 0; i < L; i++) v[i] = *reinterpret_cast<const float4*>(t + (at ^ ((uint32_t)(s0 + i) * jsb)));
#pragma unroll
                for (int i = 0; i < L; i++) {
                  C2 u[H];
                  unpack<C2, H>(v[i], u);
#pragma unroll
                  for (int q = 0; q < H; q++) {
                    const int g = (s0 + i) * H + q;
                    const C2 x = sw ? u[H - 1 - q] : u[q];
                    ar[g] = fma_(f.c, x.x, ar[g]);
                    ai[g] = fma_(f.c, x.y, ai[g]);
                  }
                }
              }
            }
            return;
          }
#pragma unroll 1
          for (; k + U <= end; k += U) some(std::integral_constant<int, U>{}, k);
          if (U > 2 && k + 2 <= end) {
            some(std::integral_constant<int, 2>{}, k);
            k += 2;
          }
          if (U > 1 && k < end) some(std::integral_constant<int, 1>{}, k);
        };
        // one slot's partner amplitudes at place `off`
        auto partner = [&](const unsigned char* t, uint32_t off, int s, bool sw, C2 (&u)[H]) {
          const uint32_t at = (jb ^ (off & ~15u)) ^ ((uint32_t)s * jsb);
          C2 v[H];
          unpack<C2, H>(*reinterpret_cast<const float4*>(t + at), v);
#pragma unroll
          for (int q = 0; q < H; q++) u[q] = sw ? v[H - 1 - q] : v[q];
        };
        // hops [k, end): 2c (= cr - cr2) where the two bits of z differ, else 0.  The thread's
        // amplitudes differ in bit 0 and in the slot bits only, so one parity per hop is computed
        // and the slots' come from the flip's slot bits (the same for all threads)
        auto hops = [&](const unsigned char* t, int k, int end) {
          const uint32_t zt = zb + (uint32_t)j0;
#pragma unroll(S >= 4 ? 1 : 2)
          for (; k < end; k++) {
            const uint32_t x = gen[k].x, off = gen[k].off;
            const R c2 = gen[k].cr - gen[k].cr2;
            const bool odd = __popc(x & zt) & 1, sw = H == 2 && (x & 1u);
            const R cA = odd ? c2 : (R)0, cB = odd ? (R)0 : c2;
            const uint32_t xs_ = (x & tmask) >> jsl;
#pragma unroll
            for (int s = 0; s < S; s++) {
              C2 u[H];
              partner(t, off, s, sw, u);
              const bool ps = __popc(xs_ & (uint32_t)s) & 1;
#pragma unroll
              for (int q = 0; q < H; q++) {
                const R cf = (ps != (sw && q)) ? cB : cA;
                ar[s * H + q] = fma_(cf, u[q].x, ar[s * H + q]);
                ai[s * H + q] = fma_(cf, u[q].y, ai[s * H + q]);
              }
            }
          }
        };
        // other products [k, end)
        auto general = [&](const unsigned char* t, int k, int end) {
#pragma unroll 1
          for (; k < end; k++) {
            const RGen<R> f = gen[k];
            const bool sw = H == 2 && (f.x & 1u);
#pragma unroll
            for (int s = 0; s < S; s++) {
              C2 u[H];
              partner(t, f.off, s, sw, u);
#pragma unroll
              for (int q = 0; q < H; q++) {
                const int g = s * H + q;
                const uint32_t zsrc = (zb + (uint32_t)(j0 + s * js + q)) ^ f.x;
                const bool n1 = __popc(f.zm & zsrc) & 1, n2 = __popc(f.zm2 & zsrc) & 1;
                const R cr = (n1 ? -f.cr : f.cr) + (n2 ? -f.cr2 : f.cr2);
                const R ci = (n1 ? -f.ci : f.ci) + (n2 ? -f.ci2 : f.ci2);
                ar[g] = fma_(cr, u[q].x, fma_(-ci, u[q].y, ar[g]));
                ai[g] = fma_(cr, u[q].y, fma_(ci, u[q].x, ai[g]));
              }
            }
          }
        };
        auto arrived = [&](uint32_t b, uint32_t parity) {
          if (!bar_wait(full0 + 8u * b, parity, &s_abort)) {
            if (!s_abort) P.slots[kSlotFault] = 1.0;
            s_abort = 1;
          }
        };
        int pk = 0, gk = 0, run = 0;
        auto runs_to = [&](const unsigned char* t, int end) {
          for (; run < end; run++) {
            const ResRun r = s_run[run];
            if (r.kind == 0) {
              plain(t, pk, r.end);
              pk = r.end;
            } else {
              if (r.kind == 1)
                hops(t, gk, r.end);
              else
                general(t, gk, r.end);
              gk = r.end;
            }
          }
        };
        if (act) runs_to(tiles, s_part[0].run_end);
        // what does not need the partners, while their tiles are on their way (owned vectors in
        // registers): the diagonal and the past's part of the corrector and the predictor
        auto code_at = [&](uint32_t j) { return tcls >= 0 ? (int)s_code[j] : 0; };
        auto diagonal = [&](uint32_t j, R (&d)[H]) {  // of the slot at j
          int code[2] = {0, 0};
#pragma unroll
          for (int q = 0; q < H; q++) {
            code[q] = code_at(j + q);
            d[q] = sc.dt[code[q]];
          }
          if (others) {
            const RSlot<R> o = other_diagonal<R>(tab, sc, s_z + par * nz, s_zm, tcls, code[0], code[1], zb + j);
#pragma unroll
            for (int q = 0; q < H; q++) d[q] += o.d[q];
          }
        };
        C2 cb[REG ? A : 1], pb[REG ? A : 1];
        R dg[REG ? A : 1];
        if (REG && act)
#pragma unroll
          for (int g = 0; g < A; g++) {
            if (g % H == 0) {
              R d[H];
              diagonal((uint32_t)(j0 + (g / H) * js), d);
#pragma unroll
              for (int q = 0; q < H; q++) dg[REG ? g + q : 0] = d[q];
            }
            if (kind == 0 || kind == 5) past(o[REG ? g / H : 0], g % H, kind, cb[REG ? g : 0], pb[REG ? g : 0]);
          }
        if (nd > 0 && !ring) {  // every partner in one go: the places name the buffers
          if (CLU)
            arrived((uint32_t)cluster_set(e), (uint32_t)(e >> 1) & 1u);
          else
            arrived(0, visit & 1u);
          if (act) runs_to(tiles, P.nruns);
        }
        uint32_t rb = ring ? q0 % (uint32_t)nbuf : 0u, ru = ring ? q0 / (uint32_t)nbuf : 0u;
        auto release = [&]() {  // this warp is done with buffer rb; on to the next ring entry
          __syncwarp();
          if (lane == 0) bar_arrive(empty0 + 8u * rb);
          if (++rb == (uint32_t)nbuf) {
            rb = 0;
            ru++;
          }
        };
        if (ring) {
          for (int p = 1; p <= nd; p++) {
            arrived(rb, ru & 1u);
            if (act) runs_to(smem + (size_t)(1u + rb) * tbytes, s_part[p].run_end);
            release();
          }
        }
        // every owner is past the products that read the own tile: it can be overwritten (in a cluster
        // the next one goes elsewhere)
        if (!CLU) asm volatile("bar.sync 1, %0;\n" ::"r"(nth) : "memory");
        R t0 = (R)0, t1 = (R)0;
        auto fetch_owned = [&](int s, Owned& w) {  // of one slot, from global memory
          const uint32_t z = zb + (uint32_t)(j0 + s * js);
          if (P.single) return;
          load(Y + z, w.y);
          if (kind == 0 || kind == 5) {
            load(F(latest) + z, w.a);
            load(F(latest - 1) + z, w.b);
            load(F(latest - 2) + z, w.c);
          }
          if (kind >= 2 && kind <= 4) load(ACC + z, w.rk);
          if (kComp && kind == 0) load(YL + z, w.yl);
        };
        const bool streamed = kStream && nq > nd;
        Owned ow[kStream ? 1 : 2];
        if (!REG && !kStream && act) fetch_owned(0, ow[0]);
#pragma unroll
        for (int s = 0; s < S; s++) {
          Owned& w = REG ? o[REG ? s : 0] : ow[kStream ? 0 : (s & 1)];
          if (streamed) {  // this slot's owned vectors from their quarter tile
            if (s % SC == 0) arrived(rb, ru & 1u);
            const C2* v = xs + (size_t)(1u + rb) * tsize + (uint32_t)(j0 + (s % SC) * js);
            load(v, w.y);
            load(v + tsize / 4, w.a);
            load(v + tsize / 2, w.b);
            load(v + 3 * (tsize / 4), w.c);
            if (s % SC == SC - 1) release();
          } else if (kStream && act) {
            fetch_owned(s, w);
          } else if (!REG && s + 1 < S && act) {
            fetch_owned(s + 1, ow[(s + 1) & 1]);
          }
          if (!act) continue;
          const uint32_t j = (uint32_t)(j0 + s * js), z0 = zb + j;
          C2 own[H], nx[H];
          R ds[H];
          load(xs_e + j, own);
          if (!REG) diagonal(j, ds);
#pragma unroll
          for (int q = 0; q < H; q++) {
            R re = ar[s * H + q], im = ai[s * H + q];
            const R d = REG ? dg[REG ? s * H + q : 0] : ds[q];
            if (d != (R)0) {  // an infinite amplitude must not make NaN of an H without diagonal
              re = fma_(d, own[q].x, re);
              im = fma_(d, own[q].y, im);
            }
            const C2 fn = C2{im, -re};  // -i (re + i im)
            C2 &y = w.y[q], &a = w.a[q], &b = w.b[q], &c = w.c[q], &rk = w.rk[q];
            if (kind == 0 || kind == 5) {
              C2 cq, pq;
              if (REG) {
                cq = cb[REG ? s * H + q : 0];
                pq = pb[REG ? s * H + q : 0];
              } else {
                past(w, q, kind, cq, pq);
              }
              if (kind == 0) {  // corrector (Adams-Moulton)
                if (sizeof(R) == 8) {
                  y.x = fma_(c9, fn.x, cq.x);
                  y.y = fma_(c9, fn.y, cq.y);
                } else {  // h/24 as hi + lo: a step size rounded to FP32 would drift over the run
                  const R sx = fma_((R)9, fn.x, cq.x), sy = fma_((R)9, fn.y, cq.y);
                  const R ix = fma_(h24, sx, h24lo * sx), iy = fma_(h24, sy, h24lo * sy);
                  if (kComp) {
                    y.x = add_compensated(y.x, w.yl[q].x, ix);
                    y.y = add_compensated(y.y, w.yl[q].y, iy);
                  } else {
                    y.x += ix;
                    y.y += iy;
                  }
                }
                const R dx = y.x - own[q].x, dy = y.y - own[q].y;
                t1 = fma_(dx, dx, fma_(dy, dy, t1));
                if (last) t0 = fma_(y.x, y.x, fma_(y.y, y.y, t0));
              }
              if (sizeof(R) == 8) {  // predictor (Adams-Bashforth)
                const R cf = kind == 0 ? c64 : p55;
                nx[q] = C2{fma_(cf, fn.x, pq.x), fma_(cf, fn.y, pq.y)};
              } else {
                const R px = fma_((R)55, fn.x, pq.x), py = fma_((R)55, fn.y, pq.y);
                nx[q] = C2{y.x + fma_(h24, px, h24lo * px), y.y + fma_(h24, py, h24lo * py)};
              }
              c = b;
              b = a;
              a = fn;
            } else if (kind == 1) {
              c = b;
              b = a;
              a = fn;
              rk = fn;
              const R hh = (R)0.5 * h;
              nx[q] = C2{fma_(hh, fn.x, y.x), fma_(hh, fn.y, y.y)};
            } else if (kind == 2 || kind == 3) {
              rk.x = fma_((R)2, fn.x, rk.x);
              rk.y = fma_((R)2, fn.y, rk.y);
              const R hh = kind == 2 ? (R)0.5 * h : h;
              nx[q] = C2{fma_(hh, fn.x, y.x), fma_(hh, fn.y, y.y)};
            } else if (kind == 4) {
              const R h6 = h / (R)6;
              y.x = fma_(h6, rk.x + fn.x, y.x);
              y.y = fma_(h6, rk.y + fn.y, y.y);
              nx[q] = y;
            } else if (kind == 6) {
              nx[q] = C2{re, im};
            } else {
              t0 = fma_(own[q].x, re, fma_(own[q].y, im, t0));
              t1 = fma_(own[q].x, im, fma_(-own[q].y, re, t1));
              nx[q] = own[q];
            }
          }
          if (kind != 7 && (!CLU || last)) store(xout + z0, nx);  // partners of a cluster get it from the tile
          if (!last && !multi) store(xs_next + j, nx);
          if (!REG) {
            if (kind == 0 || kind == 5 || kind == 1) store(F(latest + 1) + z0, w.a);
            if (kind == 0 || kind == 4) store((kind == 0 ? YO : Y) + z0, w.y);
            if (kind >= 1 && kind <= 3) store(ACC + z0, w.rk);
            if (kComp && kind == 0) store(YL + z0, w.yl);
          }
        }
        // this thread's stores, before asynchronous copies read them (a cluster's copies read the tile
        // in shared memory; the wider fence waits for the global stores, 800 cycles)
        if (CLU)
          proxy_fence_shared();
        else if (!last && nq > 0)
          proxy_fence();
        red0 += (RED)t0;
        red1 += (RED)t1;
        q0 += (uint32_t)nq;
        if (!last && multi) cta_sync();  // published before the next tile
      }
      if (kind == 0 || kind == 7) {
        s_red[(size_t)par * nth + tid] = red1;
        if (last) final0 = red0;
      }
      if (kind == 0 || kind == 5 || kind == 1) latest++;
      if (last) break;
      cta_sync();  // this CTA's part of xout is stored, the next coefficients are ready
      if (s_abort) break;  // uniform: the results are invalid and reported so
      xin = xout;
      xout = xout == XA ? XO : XA;
    }
    if (REG && act && !P.single) {  // the owned vectors back to global memory
#pragma unroll
      for (int s = 0; s < S; s++) {
        const uint32_t z = (cta << P.t) + (uint32_t)(j0 + s * js);
        if (E > P.hist) store((P.n_pec ? YO : Y) + z, o[s].y);
        if (latest > first_latest) store(F(latest) + z, o[s].a);
        if (latest > first_latest + 1) store(F(latest - 1) + z, o[s].b);
        if (latest > first_latest + 2) store(F(latest - 2) + z, o[s].c);
        if (kComp && P.n_pec) store(YL + z, o[s].yl);
      }
    }
    if (PEC || P.single == 7) {
      all_sync();  // the sums of the evaluation before the last are done: its place is free
      s_red[(size_t)(E & 1) * nth + tid] = final0;
      all_sync();
    }
  } else {
    // evaluation e's reductions over the CTA: FP64 sums in a fixed order, eight per evaluation
    // (the eight are added after the last one)
    auto lane_sums = [&](const RED* r, double* out) {
      double v = 0.0;
      for (int i = lane; i < nth; i += 32) v += (double)r[i];
      v += __shfl_down_sync(0xffffffffu, v, 16);
      v += __shfl_down_sync(0xffffffffu, v, 8);
      if (lane < 8) out[lane] = v;
    };
    double ident[3] = {tab->ident[0], tab->ident[1], tab->ident[2]};
    const double tscale = tcls >= 0 ? tab->classes[tcls].scale : 0.0;
    const int tgroup = tcls >= 0 ? tab->classes[tcls].group : 0;
    auto prepare = [&](int e) {  // coefficients of evaluation e
      const int par = e & 1;
      if (svc == 0) coefficients<R>(P, s_w + 3 * e, s_base, s_pl + par * np, s_gen + par * ng);
      if (svc == 1) diagonal_of<R>(P, s_w + 3 * e, s_z + par * nz, s_sc + par, ident, nz, ncls, tscale, tgroup);
    };
    prepare(0);
    const C2* xin = src0;
    for (int e = 0; e < E; e++) {
      const bool last = e == E - 1;
      for (uint32_t tile = cta; tile < ntiles; tile += G) {
        if (e == 0 || multi) {
          if (multi) cta_sync();
          cta_sync();
        }
        if (CLU && svc == 3) {
          if (e == 0) {
            copy_in(tile, xin, e, latest, q0);
          } else {  // the own tile to the partners
            const uint32_t k = (uint32_t)cluster_set(e), bb = full0 + 8u * k;
            const C2* const set = xs + (size_t)(k * (1u + (uint32_t)nd)) * tsize;
            if (lane == 0) expect(bb, (uint32_t)nd * tbytes);
            for (int p = lane; p < nd; p += 32)
              tile_push(saddr(set + (size_t)(1 + p) * tsize), saddr(set), tbytes, bb, cta ^ s_part[p + 1].hi);
            __syncwarp();
          }
        } else if (svc == 3 && nq > 0) {
          copy_in(tile, xin, e, latest, q0);
        }
        q0 += (uint32_t)nq;
        if (tile == cta) {
          if (!last) prepare(e + 1);
          if (PEC && svc == 2 && e > 0) lane_sums(s_red + (size_t)((e - 1) & 1) * nth, s_lane + 8 * (e - 1));
        }
        if (!last && multi) {
          cta_sync();
          if (svc == 3 && lane == 0) flag_release(P.flags + kResFlagStride * tile, (unsigned)(e + 1));
        }
      }
      const int kind = PEC ? 0 : kind_of(P, e);
      if (kind == 0 || kind == 5 || kind == 1) latest++;
      if (last) break;
      cta_sync();
      if (s_abort) break;
      if (!CLU && !multi && svc == 3 && lane == 0 && nd > 0) flag_release(P.flags + kResFlagStride * cta, (unsigned)(e + 1));
      xin = e & 1 ? XO : XA;
    }
    if (s_abort && svc == 3 && !CLU) copies_land();
    if (PEC || P.single == 7) {
      all_sync();
      all_sync();  // the last reductions are there
      if (svc == 2) {
        lane_sums(s_red + (size_t)((E - 1) & 1) * nth, s_lane + 8 * (E - 1));
        lane_sums(s_red + (size_t)(E & 1) * nth, s_lane + 8 * E);
      }
    }
  }
  const bool reduced = P.n_pec > 0 || P.single == 7;
  if (CLU) {
    // No CTA leaves while a push into or out of its shared memory is under way.  At a normal end every push
    // has been waited for; to a CTA that gave up one may still come, so that CTA waits once none is issued
    // any more, and all of them for it.
    cluster_sync();
    if (s_abort && svc == 3) copies_land();
    cluster_sync();
  }
  if (P.single == 6) return;
  __syncthreads();
  if (reduced) {
    for (int e = tid >> 5; e <= E; e += (int)blockDim.x >> 5) {
      double v = 0.0;
      if (lane == 0) {
        for (int k = 0; k < 8; k++) v += s_lane[8 * e + k];
        P.partials[(size_t)e * G + cta] = v;
      }
    }
  }
  // the last CTA sums the CTAs' partials in CTA order and clears the flags for the next launch
  int& s_last = sh.last;
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    s_last = atomicAdd(P.ticket, 1u) == G - 1 ? 1 : 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (reduced) {
    for (int e = tid >> 5; e <= E; e += (int)blockDim.x >> 5) {
      double v = 0.0;
      for (uint32_t i = lane; i < G; i += 32) v += __ldcg(&P.partials[(size_t)e * G + i]);
      v = warp_sum(v);
      if (lane == 0) s_err[e] = (e < E && P.single == 0) ? (19.0 / 270.0) * sqrt(v) : v;
    }
    __syncthreads();
    if (tid == 0) {
      if (P.single == 7) {
        P.slots[kSlotDot] = s_err[E];
        P.slots[kSlotDotIm] = s_err[0];
      } else {
        double m = inst ? inst->max_err : P.slots[kSlotMaxErr];
        for (int e = 0; e < E; e++)
          if (!(s_err[e] <= m)) m = s_err[e];  // NaN propagates
        (inst ? inst->norm2 : P.slots[kSlotNorm2]) = s_err[E];
        (inst ? inst->max_err : P.slots[kSlotMaxErr]) = m;
        (inst ? inst->last_err : P.slots[kSlotLastErr]) = s_err[E - 1];
        if (inst) {  // every CTA of the member has read its step count: on to the next steps
          inst->step += E;
          if (E & 1) {
            void* const v = inst->vec[kVecP];
            inst->vec[kVecP] = inst->vec[kVecQ];
            inst->vec[kVecQ] = v;
          }
        }
      }
    }
  }
  for (uint32_t i = tid; i < ntiles; i += blockDim.x) P.flags[kResFlagStride * i] = 0u;
  if (tid == 0) *P.ticket = 0u;
}

template <typename R, int S, bool REG, bool PEC, bool COMP>
__global__ void __launch_bounds__(owners(S) + kService, 1) k_resident(const __grid_constant__ ResParams P) {
  resident_body<R, S, REG, PEC, COMP, false>(P, blockIdx.x, gridDim.x, nullptr);
}

template <typename R, bool PEC, bool COMP>
__global__ void __launch_bounds__(kResMaxThreads + kService, 1) k_resident_cluster(const __grid_constant__ ResParams P) {
  resident_body<R, 1, true, PEC, COMP, true>(P, blockIdx.x, gridDim.x, nullptr);
}

// Predictor-corrector steps of many states in one launch: a CTA is one tile of one batch member,
// and only the CTAs of a member exchange anything.  Weights come from the member's polynomials
// (the expression of the host side).  A step of 24 complex64 members of 12 to 18 qubits (207 tiles
// of 2^13) takes 53 us in three waves on tiles of 2^12; one launch per layout level over all tiles
// took 93 us.
template <typename R, int S>
__global__ void __launch_bounds__(owners(S) + kService, 1) k_resident_batch(const __grid_constant__ ResBatch B) {
  __shared__ ResParams P;
  int m = 0;
  while (m + 1 < B.count && B.first[m + 1] <= blockIdx.x) m++;
  BatchInst* const I = B.insts + B.slot[m];
  const int64_t step = I->step, left = I->nsteps - step;
  if (left <= 0) return;  // finished: all its CTAs leave
  const int E = left < (int64_t)B.evals ? (int)left : B.evals;
  if (threadIdx.x == 0) {
    const ResArea* const A = reinterpret_cast<const ResArea*>(reinterpret_cast<const char*>(I->tab) + B.area);
    const ResMember M = A->member;
    P.tab = I->tab;
    P.rt = &A->batch;
    P.n = M.n;
    P.t = M.t;
    P.np = M.np;
    P.ng = M.ng;
    P.npart = M.npart;
    P.nbuf = M.nbuf;
    P.nruns = M.nruns;
    P.ncode = M.ncode;
    P.evals = P.n_pec = E;
    P.n_rk = P.hist = P.single = 0;
    P.step0 = (int)(step & 3) + (step >= 4 ? 4 : 0);
    P.wdev = nullptr;
    P.wstride = 0;
    P.h = I->h;
    P.dcode = I->dcode;
    P.src = I->vec[kVecP];
    P.xout[0] = I->vec[kVecQ];
    P.xout[1] = I->vec[kVecP];
    P.y = P.yout = I->vec[kVecY];
    for (int k = 0; k < 4; k++) P.f[k] = I->vec[kVecF0 + k];
    P.acc = P.ylo = nullptr;
    P.flags = M.flags;
    P.ticket = M.ticket;
    P.partials = M.partials;
    P.slots = M.slots;
  }
  for (int k = threadIdx.x; k < 3 * E; k += blockDim.x) {
    const double tau = (double)(step + k / 3 + 1) * I->h / I->T;
    const double s = I->s_kind == 1 ? tau * tau * (3.0 - 2.0 * tau) : tau;
    const double* const c = I->poly[k % 3];
    P.w[k] = ((c[3] * s + c[2]) * s + c[1]) * s + c[0];
  }
  __syncthreads();
  resident_body<R, S, (S <= 2), true, false, false>(P, blockIdx.x - B.first[m], 1u << (P.n - P.t), I);
}

template <typename R, int S, bool REG, bool PEC, bool COMP>
cudaError_t launch_t(const ResParams& p, int nth, int max_grid, int n_z, cudaStream_t s) {
  const size_t smem = ResSmem<R>(1u << p.t, p.nbuf, p.np, p.ng, n_z, nth, !REG).total;
  auto kern = k_resident<R, S, REG, PEC, COMP>;
  static KernelShape shape;
  cudaError_t e = shape.allow(kern, smem);
  if (e != cudaSuccess) return e;
  int grid = 1 << (p.n - p.t);
  if (grid > max_grid) grid = max_grid;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // CTAs that wait on one another are resident together
  attr[0].val.cooperative = 1;
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(nth + kService);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = p.evals > 1 && grid > 1 ? 1 : 0;
  e = cudaLaunchKernelEx(&cfg, kern, p);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename R, int S, bool REG>
cudaError_t launch_c(const ResParams& p, int nth, int max_grid, int n_z, cudaStream_t s) {
  if (p.n_pec == 0) return launch_t<R, S, REG, false, false>(p, nth, max_grid, n_z, s);
  return p.ylo ? launch_t<R, S, REG, true, sizeof(R) == 4>(p, nth, max_grid, n_z, s)
               : launch_t<R, S, REG, true, false>(p, nth, max_grid, n_z, s);
}

// One cluster of 2^(n - t) CTAs.  p.nbuf: two sets of partner buffers.
template <typename R, bool PEC, bool COMP>
cudaError_t launch_cluster_t(const ResParams& p, int nth, int n_z, int* fits, cudaStream_t s) {
  const size_t smem = ResSmem<R>(1u << p.t, p.nbuf, p.np, p.ng, n_z, nth, false).total;
  auto kern = k_resident_cluster<R, PEC, COMP>;
  static KernelShape shape;
  cudaError_t e = shape.allow(kern, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1u << (p.n - p.t);
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(1u << (p.n - p.t));
  cfg.blockDim = dim3(nth + kService);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (*fits < 0) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    int clusters = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg);
    if (e != cudaSuccess) return e;
    *fits = clusters > 0 ? 1 : 0;
  }
  if (*fits == 0) return cudaErrorNotSupported;
  e = cudaLaunchKernelEx(&cfg, kern, p);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename R>
cudaError_t launch_cluster_r(const ResParams& p, int nth, int n_z, int* fits, cudaStream_t s) {
  if (p.n_pec == 0) return launch_cluster_t<R, false, false>(p, nth, n_z, fits, s);
  return p.ylo ? launch_cluster_t<R, true, sizeof(R) == 4>(p, nth, n_z, fits + 2, s)
               : launch_cluster_t<R, true, false>(p, nth, n_z, fits + 1, s);
}

template <typename R>
cudaError_t launch_r(const ResParams& p, int slots, int nth, int max_grid, int n_z, cudaStream_t s) {
  const bool reg = (1 << (p.n - p.t)) <= max_grid;
  switch (slots) {
    case 1: return reg ? launch_c<R, 1, true>(p, nth, max_grid, n_z, s) : launch_c<R, 1, false>(p, nth, max_grid, n_z, s);
    case 2: return reg ? launch_c<R, 2, true>(p, nth, max_grid, n_z, s) : launch_c<R, 2, false>(p, nth, max_grid, n_z, s);
    case 8: return launch_c<R, 8, false>(p, nth, max_grid, n_z, s);
    case 16: return launch_c<R, 16, false>(p, nth, max_grid, n_z, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

size_t resident_smem_bytes(int prec, int t, int nbuf, int np, int ng, int n_z, int nth, bool reg) {
  const uint32_t tsize = 1u << t;
  return prec == 0 ? ResSmem<double>(tsize, nbuf, np, ng, n_z, nth, !reg).total
                   : ResSmem<float>(tsize, nbuf, np, ng, n_z, nth, !reg).total;
}

template <typename R, int S>
static cudaError_t launch_batch_s(const ResBatch& b, int ctas, size_t smem, cudaStream_t s) {
  auto kern = k_resident_batch<R, S>;
  static KernelShape shape;
  cudaError_t e = shape.allow(kern, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(owners(S) + kService);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, b);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename R>
static cudaError_t launch_batch_r(const ResBatch& b, int slots, int ctas, size_t smem, cudaStream_t s) {
  switch (slots) {
    case 1: return launch_batch_s<R, 1>(b, ctas, smem, s);
    case 2: return launch_batch_s<R, 2>(b, ctas, smem, s);
    case 8: return launch_batch_s<R, 8>(b, ctas, smem, s);
    case 16: return launch_batch_s<R, 16>(b, ctas, smem, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_resident_batch(int prec, const ResBatch& b, int slots, int ctas, size_t smem, cudaStream_t s) {
  return prec == 0 ? launch_batch_r<double>(b, slots, ctas, smem, s) : launch_batch_r<float>(b, slots, ctas, smem, s);
}

cudaError_t launch_resident(int prec, const ResParams& p, int slots, int nth, int max_grid, int n_z, cudaStream_t s) {
  return prec == 0 ? launch_r<double>(p, slots, nth, max_grid, n_z, s) : launch_r<float>(p, slots, nth, max_grid, n_z, s);
}

cudaError_t launch_resident_cluster(int prec, const ResParams& p, int nth, int n_z, int (&fits)[3], cudaStream_t s) {
  return prec == 0 ? launch_cluster_r<double>(p, nth, n_z, fits, s) : launch_cluster_r<float>(p, nth, n_z, fits, s);
}

}  // namespace aqc
