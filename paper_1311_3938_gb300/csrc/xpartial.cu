// Layout passes whose products are all X strings with real coefficients (the driver term of Eq. Hix
// and the XX couplings of the nonlinear path) or hops X_iX_j + Y_iY_j (Eq. Hixy), complex64 only:
//   r(z) = q(z) + [d(z) psi(z)] + sum_k c_k [hop_k: bits i_k, j_k of z differ] psi(z ^ x_k)
// for every z of the tile (gather form of the per-qubit action, Sec. I.A), then r is stored as a
// partial sum, or the contiguous layout's pass finishes the evaluation: the fused
// predictor-corrector step, a Runge-Kutta stage, the derivative or the energy.
//
// GB300 structure: one CTA of 512 threads per SM, persistent over tiles.  The 64 KiB source
// tile (2^13 amplitudes) is brought into shared memory by one TMA tensor copy
// (cp.async.bulk.tensor, 4-D map: chunk, gap bits, tile rows, top bits; the contiguous layout's by one
// plain bulk copy, with its 8 KiB of clause bytes) into one of two buffers, completion tracked by an
// mbarrier, so the next tile streams in while this one is computed.  Each thread holds 16 amplitudes
// in registers: pairs (tile bit 0) at 8 positions spanning tile bits 6..8.  Products flipping only
// bits 6..8 are register permutations; all others inside the tile read one 16-byte shared-memory
// vector per pair, at one base address plus immediate offsets.  Products that no layout holds
// read their partner from memory, one 16-byte vector per pair, in the pass that runs first.  The
// partial sum and the other vectors of a pass stream through registers, those of the epilogue one
// pair ahead.
//
// The step keeps y out of memory: with D1 = f_{n+1} - f_n, D2 = f_n - f_{n-1}, ... it forms
//   p_{n+2} = p_{n+1} + h/24 (24 f_{n+1} + 40 D1 - 55 D2 + 36 D3 - 9 D4)
// (corrector and predictor in one), and y_{n+1} = p_{n+1} + h/24 9 (D1 - 3 D2 + 3 D3 - D4) for the
// error estimate; y is stored by the last step of a call only.  Eight vectors move instead of nine,
// and the state is rounded once per step, after a sum whose large terms cancelled in differences.
//
// Measured (GB300): every pass of 28 qubits runs at the copy rate of 6.7 TB/s: partial passes 0.65 and
// 0.90 ms, the step 2.59 ms (17.4 GB; as k_apply with y in memory 2.83 ms); at 23 qubits the step
// 112 -> 96 us, the XY step of 24 qubits (78 hops, the catalyst's class) 486 -> 281 us, the last pass of
// H psi at 26 qubits 403 -> 289 us, the XY pass with products that no layout holds 178 -> 98 us (three
// layouts; 260 us where it stands for two of them).
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "aqc_internal.h"
#include "kernel_shape.h"

namespace aqc {

namespace {

constexpr int kXThreads = 512;
constexpr uint32_t kXTileBytes = (1u << kXTileBits) * 8u;  // complex64 tile
constexpr uint32_t kXRegMask = 0x1c0u;                        // tile bits 6..8: register positions
constexpr uint32_t kXWaitPolls = 1u << 24;                     // mbarrier polls before giving up

struct XFlip {
  uint32_t lx;
  float c;
  uint32_t par;  // hops: the flip mask, whose bits must differ in z; 0 for X strings
  uint32_t pad;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n"
      " .reg .pred p;\n"
      " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(bar), "r"(phase)
      : "memory");
  return ok != 0u;
}

// bounded wait for phase `phase` of the mbarrier; false if it did not complete
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t phase) {
  for (uint32_t i = 0; i < kXWaitPolls; i++)
    if (mbar_try_wait(bar, phase)) return true;
  return false;
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2,
                                            int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2,
                                            int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(bar)
      : "memory");
}

// contiguous bytes (16-byte aligned on both sides)
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst), "l"(src),
      "r"(bytes), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void fma4(float4& a, float c, const float4& g) {
  a.x = fmaf(c, g.x, a.x);
  a.y = fmaf(c, g.y, a.y);
  a.z = fmaf(c, g.z, a.z);
  a.w = fmaf(c, g.w, a.w);
}

__device__ __forceinline__ float4 swap_pair(const float4& g) { return make_float4(g.z, g.w, g.x, g.y); }

// products flipping register positions only: acc[r] += c * own[r ^ RB]
template <int RB>
__device__ __forceinline__ void reg_flip(float c, const float4 (&own)[8], float4 (&acc)[8]) {
#pragma unroll
  for (int r = 0; r < 8; r++) fma4(acc[r], c, own[r ^ RB]);
}

// other products: acc[r] += c * tile[(jw ^ sx) | ((r ^ RB) << 6)], row = tile + (jw ^ (sx & ~1)) * 8;
// SW: the flip includes the pair bit (tile bit 0), so the two amplitudes of a pair trade places
template <int RB, bool SW>
__device__ __forceinline__ void smem_flip(float c, const unsigned char* row, float4 (&acc)[8]) {
#pragma unroll
  for (int r = 0; r < 8; r++) {
    const float4 g = *reinterpret_cast<const float4*>(row + ((r ^ RB) << 9));
    fma4(acc[r], c, SW ? swap_pair(g) : g);
  }
}

// products flipping register positions and the pair bit: acc[r] += c * own[r ^ RB], its amplitudes swapped
template <int RB>
__device__ __forceinline__ void reg_flip_swap(float c, const float4 (&own)[8], float4 (&acc)[8]) {
#pragma unroll
  for (int r = 0; r < 8; r++) fma4(acc[r], c, swap_pair(own[r ^ RB]));
}

// Hops: 2c at output amplitudes whose two flipped bits differ, else 0.  Where the bits lie fixes the
// parity of a thread's amplitudes relative to its first one, and the half whose coefficient is zero
// is not read: with one register bit (RB) a thread needs four of its eight partner pairs, and which
// four is an offset of its first address; with no register bit all eight or none; with two of the
// thread's own bits (two register bits, or one and the pair bit) nothing from shared memory.  Only the
// pair bit beside a lane's or a warp's bit reads both amplitudes of every pair for one of them (8-byte
// loads at this stride conflict two ways).  XY path, n = 24, 32 steps and start-up: 24.0 -> 23.6 ms (22
// since the diagonal takes classes once per thread); the step pass keeps shared memory's pipe 46% busy
// and issue slots 42%, the one before it issue slots 51%.
// cA is the coefficient at the parity of the thread's first amplitude, cB at the opposite one.
__device__ __forceinline__ void hop_pair(float c0, float c1, const float4& g, float4& a) {
  a.x = fmaf(c0, g.x, a.x);
  a.y = fmaf(c0, g.y, a.y);
  a.z = fmaf(c1, g.z, a.z);
  a.w = fmaf(c1, g.w, a.w);
}
// one register bit; `needed` = the address of the partner rows with a coefficient, r without bit RB
template <int RB>
__device__ __forceinline__ void smem_hop_half(float cA, float cB, const unsigned char* needed, float4 (&acc)[8]) {
#pragma unroll
  for (int r = 0; r < 8; r++)
    if ((r & RB) == 0) {
      const float4 g = *reinterpret_cast<const float4*>(needed + (r << 9));
      fma4(acc[r], cA, g);
      fma4(acc[r | RB], cB, g);
    }
}
// the pair bit and a bit outside the thread
__device__ __forceinline__ void smem_hop_swap(float cA, float cB, const unsigned char* row, float4 (&acc)[8]) {
#pragma unroll
  for (int r = 0; r < 8; r++)
    hop_pair(cA, cB, swap_pair(*reinterpret_cast<const float4*>(row + (r << 9))), acc[r]);
}
// two register bits
template <int RB>
__device__ __forceinline__ void reg_hop(float cA, float cB, const float4 (&own)[8], float4 (&acc)[8]) {
#pragma unroll
  for (int r = 0; r < 8; r++) fma4(acc[r], (((r & RB) & ((r & RB) - 1)) == 0 && (r & RB) != 0) ? cB : cA, own[r ^ RB]);
}
// one register bit and the pair bit
template <int RB>
__device__ __forceinline__ void reg_hop_swap(float cA, float cB, const float4 (&own)[8], float4 (&acc)[8]) {
#pragma unroll
  for (int r = 0; r < 8; r++) {
    const bool p = (r & RB) != 0;
    hop_pair(p ? cB : cA, p ? cA : cB, swap_pair(own[r ^ RB]), acc[r]);
  }
}

__device__ __forceinline__ double weight_of(const XParams& P, int g) {
  if (P.wdev) return P.wdev[g];
  return g == 0 ? P.w[0] : (g == 1 ? P.w[1] : P.w[2]);
}

struct XSmem {  // [pad to 1 KiB][tile 0][tile 1][clause bytes 0, 1][flips][Z strings][reduction][2 mbarriers]
  size_t code, flips, z, red, bar, total;
  __host__ __device__ XSmem(int n_flips, int n_z, bool codes) {
    code = 2 * (size_t)kXTileBytes;
    flips = code + (codes ? 2u << kXTileBits : 0u);
    z = (flips + (size_t)n_flips * sizeof(XFlip) + 15) & ~(size_t)15;
    red = (z + (size_t)n_z * sizeof(float2) + 15) & ~(size_t)15;
    bar = red + 2 * (kXThreads / 32) * sizeof(double);
    total = bar + 16 + 1024;
  }
};

// Clause classes other than the byte table's and Z strings (XY path: the catalyst; Ising couplings), for
// a thread's 16 amplitudes: index zj, its pair bit and bits 6..8.  Each class, clause and string is taken
// once for all of them, a string by one parity and the signs of those four bits.  (One amplitude at a time
// 120 strings made a step at n = 24 take 1.59 ms; three layout passes with this part in the one of k_apply
// took 1.26.)
__device__ __forceinline__ void x_other_diagonal(const XParams& P, const float2* s_z, int nz, const int (&code)[16],
                                                 uint32_t zj, float (&d)[16]) {
  const DevTables* tab = P.tab;
  const int tcls = P.dcode ? tab->table_class : -1;
#pragma unroll
  for (int i = 0; i < 16; i++) d[i] = 0.f;
  for (int cc = 0; cc < tab->n_classes; cc++) {
    if (cc == tcls) continue;
    const DevClass cl = tab->classes[cc];
    const bool derived = cl.derived && tcls >= 0;
    const int b = derived ? cl.dbegin : cl.begin, e = derived ? cl.dend : cl.end;
    int cnt[16];
#pragma unroll
    for (int i = 0; i < 16; i++) cnt[i] = 0;
    for (int k = b; k < e; k++) {
      const uint32_t m = tab->clause_mask[k];
#pragma unroll
      for (int i = 0; i < 16; i++) {
        const int o = 1 - __popc(m & (zj | (uint32_t)((i >> 1) << 6) | (uint32_t)(i & 1)));
        cnt[i] += cl.pen == 0 ? (o != 0) : o * o;
      }
    }
    const float w = (float)(cl.scale * weight_of(P, cl.group));
#pragma unroll
    for (int i = 0; i < 16; i++) d[i] = fmaf(w, (float)(derived ? code[i] - cnt[i] : cnt[i]), d[i]);
  }
  for (int m = 0; m < nz; m++) {
    const uint32_t zm = __float_as_uint(s_z[m].x);
    const uint32_t c = __float_as_uint(s_z[m].y) ^ ((uint32_t)__popc(zm & zj) << 31);
    const uint32_t s0 = zm << 31, s6 = (zm >> 6) << 31, s7 = (zm >> 7) << 31, s8 = (zm >> 8) << 31;
#pragma unroll
    for (int i = 0; i < 16; i++)
      d[i] += __uint_as_float(c ^ (i & 1 ? s0 : 0u) ^ (i & 2 ? s6 : 0u) ^ (i & 4 ? s7 : 0u) ^ (i & 8 ? s8 : 0u));
  }
}

// MODE as in ApplyParams.  DIAG: this pass adds the diagonal (the contiguous layout).  FAR: it reads
// the partners of products that no layout holds.  OTHERS: the diagonal has more than the byte table's
// class (kernels of their own: the part's registers would cost the others 3%).
template <int MODE, bool DIAG, bool FAR, bool OTHERS>
__global__ void __launch_bounds__(kXThreads, 1) k_tile_x(const __grid_constant__ XParams P) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  unsigned char* const buf0 = base;
  unsigned char* const buf1 = base + kXTileBytes;
  const DevTables* tab = P.tab;
  const int fb = tab->flip_begin[P.layout_index], rb = tab->flip_begin[tab->n_layouts];
  const int npl = tab->plain_count[P.layout_index];
  const int np = npl + tab->hop_count[P.layout_index];  // X strings, then hops
  const int nf = np + (FAR ? tab->n_remote : 0);
  const int nz = DIAG && OTHERS ? tab->n_z : 0;
  const XSmem M(nf, nz, DIAG && P.dcode);
  XFlip* s_f = reinterpret_cast<XFlip*>(base + M.flips);
  float2* s_z = reinterpret_cast<float2*>(base + M.z);
  double* s_red = reinterpret_cast<double*>(base + M.red);
  uint64_t* s_bar = reinterpret_cast<uint64_t*>(base + M.bar);
  const uint32_t bar0 = smem_addr(s_bar), bar1 = smem_addr(s_bar + 1);
  const uint32_t tid = threadIdx.x;
  for (int k = tid; k < nf; k += blockDim.x) {
    const DevFlip d = tab->flips[k < np ? fb + k : rb + (k - np)];
    const bool hop = k < np ? k >= npl : d.has2 != 0;  // X_iX_j + Y_iY_j: 2c where the bits differ
    s_f[k] = XFlip{k < np ? d.lx : d.x, (float)((hop ? 2.0 : 1.0) * d.coef * weight_of(P, d.group)), hop ? d.x : 0u, 0u};
  }
  for (int k = tid; k < nz; k += blockDim.x)
    s_z[k] = make_float2(__uint_as_float(tab->z[k].zm), (float)(tab->z[k].coef * weight_of(P, tab->z[k].group)));
  float dconst = 0.f, wtab = 0.f;
  if (DIAG) {
    dconst = (float)(tab->ident[0] * weight_of(P, 0) + tab->ident[1] * weight_of(P, 1) + tab->ident[2] * weight_of(P, 2));
    if (P.dcode) wtab = (float)(tab->classes[tab->table_class].scale * weight_of(P, tab->classes[tab->table_class].group));
  }
  if (tid == 0) {
    mbar_init(bar0, 1);
    mbar_init(bar1, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();

  const Layout L = P.L;
  const uint32_t gap = (uint32_t)(L.h - L.c);
  const uint32_t lane = tid & 31u, warp = tid >> 5;
  const uint32_t jw = (warp << 9) | (lane << 1);  // tile position of this thread's first pair
  uint32_t zoff[8];                                 // index offsets of the thread's 8 pairs
#pragma unroll
  for (int r = 0; r < 8; r++) zoff[r] = tile_z(L, jw | ((uint32_t)r << 6), 0u);

  const uint32_t first = blockIdx.x, stride = gridDim.x, ntiles = P.ntiles;
  // number of the tile visited t-th: with products read from memory, tiles that differ in their top
  // bits run side by side, so that a partner's lines are in L2 when they are read
  auto number = [&](uint32_t t) {
    return FAR ? ((t & ((1u << P.top_bits) - 1u)) << gap) | (t >> P.top_bits) : t;
  };
  const float2* const src = reinterpret_cast<const float2*>(P.src);
  auto issue = [&](uint32_t t, int b) {  // thread 0: copy of the t-th tile into buffer b
    const uint32_t tile = number(t);
    const int x1 = (int)(tile & ((1u << gap) - 1u)), x3 = (int)(tile >> gap);
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    const uint32_t bb = b ? bar1 : bar0, dst = smem_addr(b ? buf1 : buf0);
    if (L.w == 0) {  // contiguous
      const size_t z = (size_t)tile << kXTileBits;
      mbar_expect_tx(bb, kXTileBytes + (DIAG && P.dcode ? 1u << kXTileBits : 0u));
      bulk_load(dst, src + z, kXTileBytes, bb);
      if (DIAG && P.dcode) bulk_load(smem_addr(base + M.code + ((size_t)b << kXTileBits)), P.dcode + z, 1u << kXTileBits, bb);
    } else {
      mbar_expect_tx(bb, kXTileBytes);
      if (P.tma_rank == 5)
        tma_load_5d(dst, &P.tmap, bb, 0, 0, x1, 0, x3);
      else
        tma_load_4d(dst, &P.tmap, bb, 0, x1, 0, x3);
    }
  };
  if (tid == 0) {
    if (first < ntiles) issue(first, 0);
    if (first + stride < ntiles) issue(first + stride, 1);
  }
  const float2* const qin = reinterpret_cast<const float2*>(P.qin);
  const float hh = (float)P.h;
  const double e24 = P.h / 24.0;
  const float h24 = (float)e24, h24lo = (float)(e24 - (double)h24);  // a step size rounded to FP32 would drift
  double red0 = 0.0, red1 = 0.0;
  uint32_t k = 0;
  for (uint32_t t_ = first; t_ < ntiles; t_ += stride, k++) {
    const int b = (int)(k & 1u);
    const uint32_t zb = tile_base(L, number(t_));
    const uint32_t zj = zb | zoff[0];  // index of the thread's first amplitude
    float4 acc[8];
    if (qin) {
#pragma unroll
      for (int r = 0; r < 8; r++) acc[r] = __ldcg(reinterpret_cast<const float4*>(qin + (zb + zoff[r])));
    } else {
#pragma unroll
      for (int r = 0; r < 8; r++) acc[r] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if constexpr (FAR) {
      // products that no layout holds (the pass waits on these loads): half of the pairs are added
      // while the other half's partners are on their way
      auto far_load = [&](const XFlip& f, int r0, float4 (&g)[4]) {
#pragma unroll
        for (int r = 0; r < 4; r++) {
          const uint32_t z = zb + zoff[r0 + r];
          // a pair with no coefficient in a hop is not read
          if (f.par == 0u || (f.lx & 1u) || (__popc(z & f.par) & 1u))
            g[r] = __ldcg(reinterpret_cast<const float4*>(src + (z ^ (f.lx & ~1u))));
          else
            g[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
      };
      auto far_add = [&](const XFlip& f, int r0, const float4 (&g)[4]) {
        const bool sw = (f.lx & 1u) != 0u;
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const int r = r0 + i;
          const float4 v = sw ? swap_pair(g[i]) : g[i];
          if (f.par) {
            const bool odd = (__popc((zb + zoff[r]) & f.par) & 1u) != 0u;
            const float c0 = odd ? f.c : 0.f, c1 = odd != sw ? f.c : 0.f;
            acc[r].x = fmaf(c0, v.x, acc[r].x);
            acc[r].y = fmaf(c0, v.y, acc[r].y);
            acc[r].z = fmaf(c1, v.z, acc[r].z);
            acc[r].w = fmaf(c1, v.w, acc[r].w);
          } else {
            fma4(acc[r], f.c, v);
          }
        }
      };
      float4 g0[4], g1[4];
      XFlip f = s_f[np];
      far_load(f, 0, g0);
      far_load(f, 4, g1);
      for (int kk = np; kk < nf; kk++) {
        const XFlip fn = s_f[kk + 1 < nf ? kk + 1 : kk];
        far_add(f, 0, g0);
        if (kk + 1 < nf) far_load(fn, 0, g0);
        far_add(f, 4, g1);
        if (kk + 1 < nf) far_load(fn, 4, g1);
        f = fn;
      }
    }
    const bool ok = mbar_wait(b ? bar1 : bar0, (k >> 1) & 1u);
    if (__syncthreads_or(!ok)) {  // uniform: a copy that never completed (not expected)
      if (tid == 0) P.slots[kSlotFault] = 1.0;
      break;
    }
    const unsigned char* t = b ? buf1 : buf0;
    float4 own[8];
#pragma unroll
    for (int r = 0; r < 8; r++) own[r] = *reinterpret_cast<const float4*>(t + ((jw | ((uint32_t)r << 6)) << 3));
    for (int kk = 0; kk < np; kk++) {
      const XFlip f = s_f[kk];
      const uint32_t rb = (f.lx & kXRegMask) >> 6, sx = f.lx & ~kXRegMask;
      if (f.par) {  // hop: one parity per thread (its first amplitude), the rest is fixed by RB, SW
        const bool pb = (__popc(zj & f.par) & 1u) != 0u;
        const float cA = pb ? f.c : 0.f, cB = pb ? 0.f : f.c;
        if (sx == 0u) {
          switch (rb) {
            case 3: reg_hop<3>(cA, cB, own, acc); break;
            case 5: reg_hop<5>(cA, cB, own, acc); break;
            default: reg_hop<6>(cA, cB, own, acc); break;
          }
        } else if (sx == 1u) {
          switch (rb) {
            case 1: reg_hop_swap<1>(cA, cB, own, acc); break;
            case 2: reg_hop_swap<2>(cA, cB, own, acc); break;
            default: reg_hop_swap<4>(cA, cB, own, acc); break;
          }
        } else {
          const unsigned char* row = t + ((jw ^ (sx & ~1u)) << 3);
          const unsigned char* needed = row + (pb ? rb << 9 : 0u);
          switch (rb | ((sx & 1u) ? 8u : 0u)) {
            case 0:
              if (pb) smem_flip<0, false>(f.c, row, acc);
              break;
            case 1: smem_hop_half<1>(cA, cB, needed, acc); break;
            case 2: smem_hop_half<2>(cA, cB, needed, acc); break;
            case 4: smem_hop_half<4>(cA, cB, needed, acc); break;
            default: smem_hop_swap(cA, cB, row, acc); break;
          }
        }
        continue;
      }
      if (sx == 0u) {
        switch (rb) {
          case 1: reg_flip<1>(f.c, own, acc); break;
          case 2: reg_flip<2>(f.c, own, acc); break;
          case 3: reg_flip<3>(f.c, own, acc); break;
          case 4: reg_flip<4>(f.c, own, acc); break;
          case 5: reg_flip<5>(f.c, own, acc); break;
          case 6: reg_flip<6>(f.c, own, acc); break;
          default: reg_flip<7>(f.c, own, acc); break;
        }
      } else if (sx == 1u) {
        switch (rb) {
          case 0: reg_flip_swap<0>(f.c, own, acc); break;
          case 1: reg_flip_swap<1>(f.c, own, acc); break;
          case 2: reg_flip_swap<2>(f.c, own, acc); break;
          case 3: reg_flip_swap<3>(f.c, own, acc); break;
          case 4: reg_flip_swap<4>(f.c, own, acc); break;
          case 5: reg_flip_swap<5>(f.c, own, acc); break;
          case 6: reg_flip_swap<6>(f.c, own, acc); break;
          default: reg_flip_swap<7>(f.c, own, acc); break;
        }
      } else {
        const unsigned char* row = t + ((jw ^ (sx & ~1u)) << 3);
        const bool sw = (sx & 1u) != 0u;
        switch (rb | (sw ? 8u : 0u)) {
          case 0: smem_flip<0, false>(f.c, row, acc); break;
          case 1: smem_flip<1, false>(f.c, row, acc); break;
          case 2: smem_flip<2, false>(f.c, row, acc); break;
          case 3: smem_flip<3, false>(f.c, row, acc); break;
          case 4: smem_flip<4, false>(f.c, row, acc); break;
          case 5: smem_flip<5, false>(f.c, row, acc); break;
          case 6: smem_flip<6, false>(f.c, row, acc); break;
          case 7: smem_flip<7, false>(f.c, row, acc); break;
          case 8: smem_flip<0, true>(f.c, row, acc); break;
          case 9: smem_flip<1, true>(f.c, row, acc); break;
          case 10: smem_flip<2, true>(f.c, row, acc); break;
          case 11: smem_flip<3, true>(f.c, row, acc); break;
          case 12: smem_flip<4, true>(f.c, row, acc); break;
          case 13: smem_flip<5, true>(f.c, row, acc); break;
          case 14: smem_flip<6, true>(f.c, row, acc); break;
          default: smem_flip<7, true>(f.c, row, acc); break;
        }
      }
    }
    // epilogue, one pair after the other; the vectors it reads come one pair ahead
    constexpr int NV = MODE == MODE_STEP ? 4 : (MODE == MODE_RK4 ? 2 : 0);
    float4 in[2][NV > 0 ? NV : 1];
    auto fetch = [&](int r, float4 (&v)[NV > 0 ? NV : 1]) {
      const uint32_t z = zb + zoff[r];
      if constexpr (MODE == MODE_STEP) {
#pragma unroll
        for (int i = 0; i < 4; i++) v[i] = *reinterpret_cast<const float4*>(reinterpret_cast<const float2*>(P.f[i]) + z);
      } else if constexpr (MODE == MODE_RK4) {
        v[0] = *reinterpret_cast<const float4*>(reinterpret_cast<const float2*>(P.y) + z);
        if (P.stage > 1) v[1] = *reinterpret_cast<const float4*>(reinterpret_cast<const float2*>(P.acc) + z);
      }
    };
    const uint8_t* const code = base + M.code + ((size_t)b << kXTileBits);
    auto counts = [&](int r, int& k0, int& k1) {  // cached clause counts of a pair
      k0 = k1 = 0;
      if (P.dcode) {
        const uint32_t two = *reinterpret_cast<const uint16_t*>(code + (jw | ((uint32_t)r << 6)));
        k0 = (int)(two & 0xffu);
        k1 = (int)(two >> 8);
      }
    };
    // (selects: a branch lets the warp's stores come apart, 1% of a step at 28 qubits)
    auto add_diagonal = [&](float d0, float d1, const float4& w, float4& a) {
      const bool n0 = d0 != 0.f, n1 = d1 != 0.f;
      const float4 t = make_float4(fmaf(d0, w.x, a.x), fmaf(d0, w.y, a.y), fmaf(d1, w.z, a.z), fmaf(d1, w.w, a.w));
      a = make_float4(n0 ? t.x : a.x, n0 ? t.y : a.y, n1 ? t.z : a.z, n1 ? t.w : a.w);
    };
    if constexpr (DIAG && OTHERS) {
      int k16[16];
      float od[16];
#pragma unroll
      for (int r = 0; r < 8; r++) counts(r, k16[2 * r], k16[2 * r + 1]);
      x_other_diagonal(P, s_z, nz, k16, zj, od);
#pragma unroll
      for (int r = 0; r < 8; r++)
        add_diagonal(fmaf(wtab, (float)k16[2 * r], dconst) + od[2 * r],
                     fmaf(wtab, (float)k16[2 * r + 1], dconst) + od[2 * r + 1], own[r], acc[r]);
    }
    if (NV > 0) fetch(0, in[0]);
    float t0 = 0.f, t1 = 0.f;
#pragma unroll
    for (int r = 0; r < 8; r++) {
      if (NV > 0 && r < 7) fetch(r + 1, in[(r + 1) & 1]);
      const uint32_t z = zb + zoff[r];
      float4 a = acc[r];
      const float4 w = own[r];
      if constexpr (DIAG && !OTHERS) {
        int k0, k1;
        counts(r, k0, k1);
        add_diagonal(fmaf(wtab, (float)k0, dconst), fmaf(wtab, (float)k1, dconst), w, a);
      }
      auto put = [&](void* v, const float4& x) { *reinterpret_cast<float4*>(reinterpret_cast<float2*>(v) + z) = x; };
      const float4 fn = make_float4(a.y, -a.x, a.w, -a.z);  // -i r
      if constexpr (MODE == MODE_PARTIAL) {
        put(P.qout, a);
      } else if constexpr (MODE == MODE_DERIV) {
        put(P.fout, fn);
      } else if constexpr (MODE == MODE_ENERGY) {
        t0 += (w.x * a.x + w.y * a.y) + (w.z * a.z + w.w * a.w);
        t1 += (w.x * a.y - w.y * a.x) + (w.z * a.w - w.w * a.z);
      } else if constexpr (MODE == MODE_STEP) {
        const float4(&v)[NV] = in[r & 1];  // f_n, f_{n-1}, f_{n-2}, f_{n-3}
        put(P.fout, fn);
        float4 pn, yn;
        auto one = [&](float p, float f, float f0, float f1, float f2, float f3, float& po, float& yo) {
          const float d1 = f - f0, d2 = f0 - f1, d3 = f1 - f2, d4 = f2 - f3;
          const float s = fmaf(24.f, f, fmaf(40.f, d1, fmaf(-55.f, d2, fmaf(36.f, d3, -9.f * d4))));
          const float c = 9.f * ((d1 - d4) + 3.f * (d3 - d2));
          po = p + fmaf(h24, s, h24lo * s);
          const float e = fmaf(h24, c, h24lo * c);
          yo = p + e;
          t1 = fmaf(e, e, t1);  // y - p
        };
        one(w.x, fn.x, v[0].x, v[1].x, v[2].x, v[3].x, pn.x, yn.x);
        one(w.y, fn.y, v[0].y, v[1].y, v[2].y, v[3].y, pn.y, yn.y);
        one(w.z, fn.z, v[0].z, v[1].z, v[2].z, v[3].z, pn.z, yn.z);
        one(w.w, fn.w, v[0].w, v[1].w, v[2].w, v[3].w, pn.w, yn.w);
        put(P.pout, pn);
        if (P.yout) put(P.yout, yn);
      } else if constexpr (MODE == MODE_RK4) {
        const float4 y = in[r & 1][0];
        float4 s = in[r & 1][1];
        if (P.stage == 1) {
          put(P.fout, fn);  // history f_n
          s = fn;
        } else {
          const float m = P.stage == 4 ? 1.f : 2.f;
          s = make_float4(fmaf(m, fn.x, s.x), fmaf(m, fn.y, s.y), fmaf(m, fn.z, s.z), fmaf(m, fn.w, s.w));
        }
        const float c = P.stage == 4 ? hh / 6.f : (P.stage == 3 ? hh : 0.5f * hh);
        const float4 u = P.stage == 4 ? s : fn;
        const float4 x = make_float4(fmaf(c, u.x, y.x), fmaf(c, u.y, y.y), fmaf(c, u.z, y.z), fmaf(c, u.w, y.w));
        if (P.stage < 4) put(P.acc, s);
        put(P.stage < 4 ? P.pout : P.y, x);
      }
    }
    red0 += (double)t0;
    red1 += (double)t1;
    __syncthreads();  // every read of buffer b is done: it can take the tile after next
    if (tid == 0 && t_ + 2 * stride < ntiles) issue(t_ + 2 * stride, b);
  }
  // A CTA that gave up at tile k leaves only after the copies issued for tiles k and k + 1 have
  // landed (bounded); after a normal end no copy is outstanding.
  if (tid == 0) {
    for (uint32_t kq = k; kq < k + 2u; kq++)
      if (first + kq * stride < ntiles) (void)mbar_wait((kq & 1u) ? bar1 : bar0, (kq >> 1) & 1u);
  }
  __syncthreads();
  if (MODE != MODE_STEP && MODE != MODE_ENERGY) return;
  // FP64 sums: lanes, warps and CTAs in a fixed order; the last CTA writes the result slots
  auto cta_sum = [&](double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    double s = 0.0;
    if (tid == 0)
      for (int w = 0; w < kXThreads / 32; w++) s += s_red[w];
    return s;
  };
  __shared__ int s_last;
  const double v0 = MODE == MODE_ENERGY ? cta_sum(red0) : 0.0, v1 = cta_sum(red1);
  if (tid == 0) {
    P.partials[2 * blockIdx.x] = v0;
    P.partials[2 * blockIdx.x + 1] = v1;
    __threadfence();
    s_last = atomicAdd(P.counter, 1u) == gridDim.x - 1 ? 1 : 0;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double a0 = 0.0, a1 = 0.0;
  for (uint32_t i = tid; i < gridDim.x; i += blockDim.x) {
    a0 += __ldcg(&P.partials[2 * i]);
    a1 += __ldcg(&P.partials[2 * i + 1]);
  }
  a0 = cta_sum(a0);
  a1 = cta_sum(a1);
  if (tid == 0) {
    if (MODE == MODE_ENERGY) {
      P.slots[kSlotDot] = a0;
      P.slots[kSlotDotIm] = a1;
    } else {
      const double e = (19.0 / 270.0) * sqrt(a1);
      P.slots[kSlotLastErr] = e;
      if (!(e <= P.slots[kSlotMaxErr])) P.slots[kSlotMaxErr] = e;  // NaN propagates
    }
    *P.counter = 0u;
  }
}

template <int MODE, bool DIAG, bool FAR = false, bool OTHERS = false>
cudaError_t launch_x(const XParams& p, int n_flips, int n_z, cudaStream_t s) {
  const size_t smem = XSmem(n_flips, n_z, DIAG && p.dcode).total;
  auto kern = k_tile_x<MODE, DIAG, FAR, OTHERS>;
  static KernelShape shape;
  const cudaError_t e = shape.allow(kern, smem);
  if (e != cudaSuccess) return e;
  const int g = (uint32_t)p.max_grid > p.ntiles ? (int)p.ntiles : p.max_grid;
  kern<<<g, kXThreads, smem, s>>>(p);
  return cudaGetLastError();
}

template <int MODE>
cudaError_t launch_diag(const XParams& p, int n_flips, int n_z, cudaStream_t s) {
  return p.others ? launch_x<MODE, true, false, true>(p, n_flips, n_z, s) : launch_x<MODE, true>(p, n_flips, n_z, s);
}

}  // namespace

bool tile_x_layout_ok(const Layout& L) {
  if (L.cb != 0 || L.t != kXTileBits) return false;
  // TMA box: the chunk as 2^(c+1) floats (one box row up to c = 7, else 256 x 2^(c-7)), 2^w <= 256
  // rows; or a contiguous tile
  return L.w == 0 || (L.c >= 1 && L.c <= 12 && L.w <= 8 && L.h > L.c);
}

size_t tile_x_smem_bytes(int n_flips, int n_z, bool codes) { return XSmem(n_flips, n_z, codes).total; }

cudaError_t launch_tile_x(const XParams& p, int n_flips, int n_z, cudaStream_t s) {
  if (p.with_remote && (p.mode != MODE_PARTIAL || p.with_diag)) return cudaErrorInvalidValue;
  if (!p.with_diag) {
    if (p.mode != MODE_PARTIAL) return cudaErrorInvalidValue;
    return p.with_remote ? launch_x<MODE_PARTIAL, false, true>(p, n_flips, 0, s)
                         : launch_x<MODE_PARTIAL, false>(p, n_flips, 0, s);
  }
  switch (p.mode) {
    case MODE_PARTIAL: return launch_diag<MODE_PARTIAL>(p, n_flips, n_z, s);
    case MODE_STEP: return launch_diag<MODE_STEP>(p, n_flips, n_z, s);
    case MODE_RK4: return launch_diag<MODE_RK4>(p, n_flips, n_z, s);
    case MODE_DERIV: return launch_diag<MODE_DERIV>(p, n_flips, n_z, s);
    case MODE_ENERGY: return launch_diag<MODE_ENERGY>(p, n_flips, n_z, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace aqc
