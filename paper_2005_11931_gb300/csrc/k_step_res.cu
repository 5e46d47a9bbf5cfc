// On-chip resident leapfrog: every step of a call in one cooperative launch, the fields held by the
// SMs from the first step to the last (FP32, increment form; the scheme of k_step.cu,
// arXiv:2005.11931 Sec. 2 eq. (2.1) on the Sec. 3.3 box).
//
// A grid of up to about 2000^2 nodes needs 16 bytes per node (u, v, hx, hy), and the 152 SMs hold
// 256 KB of registers, 227 KB of shared memory and 256 KB of tensor memory each.  So no step reads
// a field from memory: one CTA per SM owns a tile of 120 columns x `rows` rows and keeps it with a
// halo of 4 (128 columns, one float4 per lane; rows + 8 rows over 16 warps of R rows).  Within a CTA
// the warps exchange the first and last of their rows through shared memory once per step; after
// four steps, when the halo is used up, each CTA stores the 4-deep rim of its tile into a buffer in
// the L2 and reads its halo from its up to 8 neighbours' rims.  Each 8 bytes of a rim carry a value
// and the pass that wrote it, so the reader polls the data themselves (a flag behind a fence took
// 1.30 us per step at 64^2 with the energy instead of 1.05).
//
// What bounds it: the FP32 pipe and instruction issue (without the energy 59 warp instructions per row of
// 128 nodes and step at 8 rows per warp, 61 at 17, 33 of them FP32 arithmetic; streaming tiles through
// shared memory and register windows, as k_step_wtb.cu does, takes 100 to 176), and one exchange, about
// 2 us, per four steps.
// Measured (GB300, us per step, before and after): 769^2 with receivers 4.1 and 1.35; 1024^2 3.6 and
// 1.43, 1400^2 4.6 and 1.9, 2048^2 5.9 and 4.7; with the energy 1003 x 517 4.8 and 1.7, 1024^2 4.9 and
// 1.8, 1536^2 5.7 and 3.1, 2048^2 6.85 and 6.1.
//
// All warps run the row code in step (a barrier per step): when only neighbouring warps waited for
// each other they drifted apart, and the unrolled code of all of them no longer fitted the
// instruction cache (2048^2 18 us per step).  For the same reason there is one copy of it: boundary
// columns have coefficients 0 instead of a masked copy.
//
// Where a tile lives (rows per warp R, 16 warps of at most 128 registers):
//   narrow: u and v in registers, hx and hy in shared memory (16 KB per row of all warps);
//   wide:   u in registers, v in shared memory, hx and hy in tensor memory (16 rows x 8 columns
//           of a warp's quarter of the 32 lanes; a 17th row in shared memory).  Tensor memory is
//           used as a plain scratchpad (tcgen05.st once, tcgen05.ld per row and step).
// Wide from 5 rows per warp on: 1200^2 2.50 against 3.12 us per step with the energy, 1400^2 1.90 against
// 2.01 and 1536^2 2.28 against 3.17 without (the narrow tile spills); no difference at 2 to 4 rows.
//
// The arithmetic of a node is that of k_step_wtb.cu operation by operation, so the states equal the
// other passes' bit for bit, and the energy's terms are added up along the same chains of rows.
#include <string.h>

#include <atomic>
#include <type_traits>

#include "async_copy.cuh"
#include "stencil_common.cuh"

namespace tsu {
namespace {
using namespace dev;

constexpr int kResWarps = 16, kResThreads = kResWarps * 32;
constexpr int kResK = 4;        // steps per exchange = halo depth (one lane of four columns)
constexpr int kResOut = 120;    // output columns per strip: strip s reads 120 s - 8 .. 120 s + 119
// Energy partials are kept for kResEnergySteps steps and summed by a launch of their own
// (k_res_energy), so a longer call with the energy runs as several launches (each reads the fields
// on chip and writes them back, about 15 us for 1024 steps of 1 ms or more).
constexpr int64_t kResEnergySteps = 1024;
constexpr int kResChain = 16;  // rows of an energy chain (k_step_wtb.cu's smallest tile)
// A launch never runs longer than a fraction of a second, so that another resident launch on the
// device, whose CTAs may be placed as this one's leave, gets its SMs well inside the bound of its waits.
constexpr int64_t kResMaxSteps = 16384;

// One lane's four columns of u and v as they travel between CTAs: every 8 bytes hold a value and
// the number of the pass that wrote it, so a reader polls the data itself and no flag, fence or
// barrier stands between the store and its use.  The accesses are vectors of two 64-bit elements: an
// aligned 8-byte element is read and written whole, while of a vector of 32-bit elements the memory
// model would allow a reader to see the tag without the value.
struct alignas(16) ResItem {
  uint64_t w[8];  // value | tag << 32
};
static_assert(sizeof(ResItem) == 64, "item");

struct ResArgs {
  int32_t nx, ny;
  int64_t ld;
  float cx, cy;
  const float* hx;
  const float* hy;
  const float* u;
  const float* v;
  float* uo;
  float* vo;
  int rows, nstrips, nchunks;
  int64_t nsteps;
  double* part;  // [step][CTA] energy partials
  float2* es;    // [CTA][kResK][thread], lean tiles
  ResItem* col;  // [2][CTA][2][16 R] the first and last output lane of every row
  ResItem* row;  // [2][CTA][2][4][32] the first and last four output rows
  int* status;
  float* traces;
  int32_t nrec;
  const int* rec_off;
  const int4* rec_ent;
  PollLimit wait;
  uint32_t skew;  // added to the tags sent: 0 (test hook: a number that no reader waits for)
};

// rows r < kTmemRows of a wide tile keep their faces in tensor memory
constexpr int kTmemRows = 16;
// Wide tiles of more than 12 rows with the energy: shared memory holds the terms of one step only (a
// barrier more per step, between the chains and the next rows), the rims' staging shares their
// place, and the chains' results of a pass wait in the workspace.
constexpr bool res_lean(int R, bool ENERGY) { return ENERGY && R > 12; }
// Tiles of up to 8 rows per warp keep the terms of all the steps of a pass and add them up at its end,
// four chains at a time, while the rims travel, instead of one step behind the rows: 1024^2 1.82 against
// 1.93 us per step, 1200^2 2.30 against 2.50; at 10 rows 3.18 against 3.02.
constexpr bool res_batch(int R, bool ENERGY) { return ENERGY && R <= 8; }
template <int R, bool WIDE, bool ENERGY>
struct ResSmem {
  static constexpr bool kLean = res_lean(R, ENERGY), kBatch = res_batch(R, ENERGY);
  static constexpr int kStage = 4 * R > 32 ? 4 * R : 32;
  float4 xch[2][kResWarps][2][32];   // first and last u row of every warp, double buffered
  // energy: the terms of the last steps summed over each lane's columns, the (sum, error) of each
  // thread's chain of rows for the pass's steps, and those of each warp
  static constexpr int kEr = kBatch ? kResK : ENERGY && !kLean ? 2 : 1;
  static constexpr bool kEs = ENERGY && !kLean && !kBatch;
  alignas(16) float er[kEr][ENERGY ? kResWarps * R : 1][32];
  float2 es[kEs ? kResK : 1][kEs ? kResThreads : 1];
  float3 esw[kResK][kResWarps];
  int2 rec[kResMaxRec];              // (row << 8 | column in the tile, receiver)
  // per warp: one row of u, or the values of its first and last output lanes on their way
  float4 stage[kLean ? 1 : kResWarps][kLean ? 1 : kStage];
  uint32_t tmem;
  // narrow: [R][2] float4 per thread (hx, hy); wide: [R] v, the faces of the rows past kTmemRows
  // or else the hy row below the warp's first
  static constexpr int kField = WIDE ? R + 2 * (R > kTmemRows ? R - kTmemRows : 0) + (R > kTmemRows ? 0 : 1) : 2 * R;
  alignas(16) float4 f[kField][kResThreads];
};

__device__ __forceinline__ P4 as_p4(const float4& v) { return P4{{pk(v.x, v.y), pk(v.z, v.w)}}; }
__device__ __forceinline__ float4 as_f4(const P4& v) {
  const float2 a = upk(v.p[0]), b = upk(v.p[1]);
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float4 ldcg4(const float* g, bool ok) {
  return ok ? __ldcg(reinterpret_cast<const float4*>(g)) : make_float4(0.f, 0.f, 0.f, 0.f);
}
__device__ __forceinline__ uint64_t tagged(float x, const uint32_t tag) {
  return (uint64_t)tag << 32 | __float_as_uint(x);
}
__device__ __forceinline__ void item_put(ResItem* d, const float4& u, const float4& v, const uint32_t tag) {
  auto st = [&](int k, float x, float y) {
    asm volatile("st.volatile.global.v2.b64 [%0], {%1, %2};" ::"l"(&d->w[2 * k]), "l"(tagged(x, tag)), "l"(tagged(y, tag))
                 : "memory");
  };
  st(0, u.x, u.y);
  st(1, u.z, u.w);
  st(2, v.x, v.y);
  st(3, v.z, v.w);
}
__device__ __forceinline__ bool item_try(const ResItem* d, float4& u, float4& v, const uint32_t tag) {
  uint64_t x[8];
#pragma unroll
  for (int k = 0; k < 4; ++k)
    asm volatile("ld.volatile.global.v2.b64 {%0, %1}, [%2];"
                 : "=l"(x[2 * k]), "=l"(x[2 * k + 1])
                 : "l"(&d->w[2 * k])
                 : "memory");
  auto value = [&](int k) { return __uint_as_float((uint32_t)x[k]); };
  u = make_float4(value(0), value(1), value(2), value(3));
  v = make_float4(value(4), value(5), value(6), value(7));
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 8; ++k) ok = ok && (uint32_t)(x[k] >> 32) == tag;
  return ok;
}
// a call of its own: inlined, its registers spilled others of the steps (1800^2 with the energy 4.78 us per
// step instead of 4.09)
__device__ __noinline__ bool item_over(const PollLimit w, const uint64_t t0) { return poll_over(w, t0); }
// The item of pass `tag`, waited for with a bound (its CTA is resident: cooperative launch).  dead: a wait ran
// out, now or before; what is not there is NaN, so that no result of it looks valid.
__device__ __forceinline__ void item_get(const ResItem* d, float4& u, float4& v, const uint32_t tag, const PollLimit& w,
                                         bool& dead) {
  if (item_try(d, u, v, tag)) return;
  if (!dead) {
    const uint64_t t0 = global_ns();
    for (int it = 0; it < kPollCap; ++it) {
      if (item_try(d, u, v, tag)) return;
      if ((it & 63) == 63 && item_over(w, t0)) break;
    }
  }
  dead = true;
  const float nan = __uint_as_float(0x7fffffffu);
  u = v = make_float4(nan, nan, nan, nan);
}
// ---- tensor memory as a scratchpad: 8 columns of the warp's 32 lanes per call -------------------
struct Tm8 {
  uint32_t r[8];
};
__device__ __forceinline__ void tmem_st8(uint32_t addr, const float4& a, const float4& b) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr),
               "r"(__float_as_uint(a.x)), "r"(__float_as_uint(a.y)), "r"(__float_as_uint(a.z)),
               "r"(__float_as_uint(a.w)), "r"(__float_as_uint(b.x)), "r"(__float_as_uint(b.y)),
               "r"(__float_as_uint(b.z)), "r"(__float_as_uint(b.w))
               : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t addr, Tm8& d) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(d.r[0]), "=r"(d.r[1]), "=r"(d.r[2]), "=r"(d.r[3]), "=r"(d.r[4]), "=r"(d.r[5]), "=r"(d.r[6]),
                 "=r"(d.r[7])
               : "r"(addr)
               : "memory");
}
// wait for the load; the registers pass through so that no use of them moves above it
__device__ __forceinline__ void tmem_wait_ld(Tm8& d) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(d.r[0]), "+r"(d.r[1]), "+r"(d.r[2]), "+r"(d.r[3]), "+r"(d.r[4]), "+r"(d.r[5]), "+r"(d.r[6]),
                 "+r"(d.r[7])::"memory");
}
__device__ __forceinline__ P4 tm_p4(const Tm8& d, int o) {
  return P4{{pk(__uint_as_float(d.r[o]), __uint_as_float(d.r[o + 1])),
             pk(__uint_as_float(d.r[o + 2]), __uint_as_float(d.r[o + 3]))}};
}

// a += b, sums as three FP32 numbers: the errors of the highs go into the middles, theirs into the lows, about
// 70 bits, where the other passes add in FP64 (two numbers, 46 bits, left energies off by up to 9e-15 from the
// FP64 sums of the same chains, 64^2 to 2048^2; these by at most 6e-16, and cost 1 to 2 % more; FP64 itself
// issues a warp instruction every 64 clocks)
__device__ __forceinline__ float two_sum(float& s, const float b) {  // s += b; the error
  const float t = __fadd_rn(s, b), z = __fsub_rn(t, s);
  const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(b, z));
  s = t;
  return e;
}
__device__ __forceinline__ void sum_add(float3& a, const float3 b) {
  const float e1 = two_sum(a.x, b.x), e2 = two_sum(a.y, b.y), e3 = two_sum(a.y, e1);
  a.z = __fadd_rn(__fadd_rn(a.z, b.z), __fadd_rn(e2, e3));
}

template <int R, int RB, bool WIDE, bool ENERGY, bool REC>
__global__ void __launch_bounds__(kResThreads, 1) k_leapfrog_res(const ResArgs a) {
  using Smem = ResSmem<R, WIDE, ENERGY>;
  constexpr bool LEAN = Smem::kLean, BATCH = Smem::kBatch;
  static_assert(!LEAN || !REC, "no place to stage receivers");
  static_assert(!LEAN || sizeof(Smem::er) >= sizeof(float4) * kResWarps * Smem::kStage, "staging");
  extern __shared__ __align__(16) unsigned char res_raw[];
  Smem& sm = *reinterpret_cast<Smem*>(res_raw);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int cta = blockIdx.x, nsx = a.nstrips, ncta = gridDim.x;
  const int chunk = cta / nsx, strip = cta - chunk * nsx;
  const int c0 = strip * kResOut - 8 + 4 * lane;
  const int y0 = 1 + chunk * a.rows, y1 = min(y0 + a.rows, a.ny - 1);
  const int rw = y0 - kResK + w * R;  // this warp's first row
  const bool col_in = c0 >= 0 && c0 < a.ld;  // the whole float4 lies in the row (ld % 4 == 0)
  const bool col_out = lane >= 1 && lane <= 30 && col_in;

  uint32_t tbase = 0;
  if constexpr (WIDE) {
    if (w == 0) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&sm.tmem))
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
  }
  __syncthreads();
  // the warp's quarter of the lanes (w % 4) and its 128 columns (w / 4)
  if constexpr (WIDE) tbase = *(volatile uint32_t*)&sm.tmem + ((uint32_t)(w & 3) << 21) + (uint32_t)(w >> 2) * 128;

  // ---- the tile: rows rw .. rw + R - 1 of this warp (zeros outside the grid and past the halo)
  P4 u[R];
  [[maybe_unused]] P4 vreg[WIDE ? 1 : R] = {};
  auto row_held = [&](int r) { return rw + r >= 0 && rw + r < a.ny && rw + r < y1 + kResK; };
  auto goff = [&](int r) { return (int64_t)(rw + r) * a.ld + c0; };
  auto get_v = [&](int r) -> P4 {
    if constexpr (WIDE)
      return as_p4(sm.f[r][tid]);
    else
      return vreg[r];
  };
  auto set_v = [&](int r, const P4& x) {
    if constexpr (WIDE)
      sm.f[r][tid] = as_f4(x);
    else
      vreg[r] = x;
  };
  // Columns lo .. hi of a row.  No step masks the boundary columns or the padding (their
  // coefficients are 0), so whatever lies in the padding or in a face that borders no interior node is
  // dropped here: 0 times a NaN or an infinity would not be 0.  Bit masks, opaque to the compiler: kept
  // comparisons spilled (1800^2 with the energy 4.27 against 4.09 us per step).
  auto keep = [&](int lo, int hi) {
    uint4 m = make_uint4(0u, 0u, 0u, 0u);
    uint32_t* const e = &m.x;
#pragma unroll
    for (int k = 0; k < 4; ++k) e[k] = c0 + k >= lo && c0 + k <= hi ? 0xffffffffu : 0u;
    asm volatile("" : "+r"(m.x), "+r"(m.y), "+r"(m.z), "+r"(m.w));
    return m;
  };
  const uint4 mnode = keep(1, a.nx - 2), mface = keep(0, a.nx - 2);
  auto cols = [&](const float4& x, const uint4& m) {
    return make_float4(__uint_as_float(__float_as_uint(x.x) & m.x), __uint_as_float(__float_as_uint(x.y) & m.y),
                       __uint_as_float(__float_as_uint(x.z) & m.z), __uint_as_float(__float_as_uint(x.w) & m.w));
  };
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const bool ok = col_in && row_held(r);
    u[r] = as_p4(cols(ldcg4(a.u + goff(r), ok), mnode));
    set_v(r, as_p4(cols(ldcg4(a.v + goff(r), ok), mnode)));
    const float4 fx = cols(ldcg4(a.hx + goff(r), ok), mface);
    const float4 fy = cols(ldcg4(a.hy + goff(r), ok), mnode);
    if constexpr (WIDE) {
      if (r < kTmemRows) {
        tmem_st8(tbase + 8 * r, fx, fy);
      } else {
        sm.f[R + 2 * (r - kTmemRows)][tid] = fx;
        sm.f[R + 2 * (r - kTmemRows) + 1][tid] = fy;
      }
    } else {
      sm.f[2 * r][tid] = fx;
      sm.f[2 * r + 1][tid] = fy;
    }
  }
  if constexpr (WIDE) asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  if constexpr (WIDE && R <= kTmemRows) {
    const bool ok = col_in && rw - 1 >= 0 && rw - 1 < a.ny && rw - 1 < y1 + kResK;
    sm.f[Smem::kField - 1][tid] = cols(ldcg4(a.hy + goff(-1), ok), mnode);
  }
  float4* const stage = (LEAN ? reinterpret_cast<float4*>(&sm.er[0][0][0]) : &sm.stage[0][0]) + w * Smem::kStage;
  // receivers of the tile's own nodes; rec_rows: this warp's rows that hold some
  [[maybe_unused]] int nrec = 0;
  [[maybe_unused]] uint32_t rec_rows = 0;
  if constexpr (REC) {
    // the table's tile order: the two outer strips first, then chunk by chunk
    const int t = nsx < 3 ? cta
                  : strip == 0 ? 2 * chunk
                  : strip == nsx - 1 ? 2 * chunk + 1 : 2 * a.nchunks + chunk * (nsx - 2) + strip - 1;
    const int lo = a.rec_off[t];
    nrec = min(a.rec_off[t + 1] - lo, kResMaxRec);
    for (int q = tid; q < nrec; q += kResThreads) {
      const int4 e = a.rec_ent[lo + q];
      sm.rec[q] = make_int2((e.x << 8) | (e.y - (strip * kResOut - 8)), e.z);
    }
    __syncthreads();
    for (int q = 0; q < nrec; ++q) {
      const int r = (sm.rec[q].x >> 8) - rw;
      if (r >= 0 && r < R) rec_rows |= 1u << r;
    }
  }
  // rows whose nodes are interior, and those this tile owns; warps with nothing to mask or record
  // run a copy of the row code without the tests
  uint32_t in_rows = 0, own_rows = 0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (rw + r >= 1 && rw + r <= a.ny - 2) in_rows |= 1u << r;
    if (rw + r >= y0 && rw + r < y1) own_rows |= 1u << r;
  }
  // rows it sends to the chunks above and below, and rows it receives from them (a neighbour's row
  // inside the grid; the boundary rows and what lies beyond stay as loaded)
  uint32_t rim_rows = 0, halo_rows = 0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int j = rw + r;
    if ((own_rows >> r) & 1u)
      rim_rows |= ((chunk > 0 && j < y0 + kResK) || (chunk + 1 < a.nchunks && j >= y1 - kResK)) ? 1u << r : 0u;
    else if ((in_rows >> r) & 1u)
      halo_rows |= ((j < y0 && j >= y0 - kResK) || (j >= y1 && j < y1 + kResK)) ? 1u << r : 0u;
  }
  constexpr uint32_t all_rows = R == 32 ? 0xffffffffu : (1u << R) - 1u;
  // -tau^2/dx^2 and -tau^2/dy^2 of the lane's columns, 0 on boundary columns and beyond, whose nodes
  // so keep the v = 0 and u = 0 they were loaded with (the results are masked once more when they are stored)
  bool ncol[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) ncol[e] = c0 + e >= 1 && c0 + e <= a.nx - 2;
  f2x ncx2[2], ncy2[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    ncx2[q] = pk(ncol[2 * q] ? -a.cx : 0.f, ncol[2 * q + 1] ? -a.cx : 0.f);
    ncy2[q] = pk(ncol[2 * q] ? -a.cy : 0.f, ncol[2 * q + 1] ? -a.cy : 0.f);
  }

  const int npass = (int)((a.nsteps + kResK - 1) / kResK);
  bool dead = false;
  // this CTA's rims and those it reads (the neighbours exist where the halo lies in the grid)
  const int T = kResWarps * R;
  auto col_rim = [&](int q, int c, int side) { return a.col + (((int64_t)q * ncta + c) * 2 + side) * T + w * R; };
  auto row_rim = [&](int q, int c, int side, int k) {
    return a.row + ((((int64_t)q * ncta + c) * 2 + side) * kResK + k) * 32;
  };
  const bool has_l = strip > 0, has_r = strip + 1 < nsx;

  // The energy terms of a step (one per row and lane: the sum over the lane's four columns) are added
  // up along the chains that k_step_wtb.cu's tiles of 16 rows have: same rows, same order, same
  // compensation, so the energies agree with the other passes' (a compensated FP32 sum of terms of
  // both signs is off by about 1e-9, and by another 1e-9 in any other order).  Thread 32 c + l takes
  // chunk c of lane l, one step behind the rows.
  [[maybe_unused]] auto chain = [&](int s) {
    float es = 0.f, ec = 0.f;
    const int r0 = kResK + kResChain * w, r1 = min(r0 + kResChain, kResK + y1 - y0);
    if (col_out) {
#pragma unroll 4
      for (int r = r0; r < r1; ++r) {
        const float y = sm.er[s % Smem::kEr][r][lane] - ec;
        const float sum = es + y;
        ec = (sum - es) - y;
        es = sum;
      }
    }
    if constexpr (LEAN)
      a.es[((int64_t)cta * kResK + s) * kResThreads + tid] = make_float2(es, -ec);
    else if constexpr (Smem::kEs)
      sm.es[s][tid] = make_float2(es, -ec);
  };

  int buf = 0;
  for (int p = 0; p < npass; ++p) {
    const int ns = (int)min((int64_t)kResK, a.nsteps - (int64_t)p * kResK);
    for (int s = 0; s < ns; ++s) {
      sm.xch[buf][w][0][lane] = as_f4(u[0]);
      sm.xch[buf][w][1][lane] = as_f4(u[R - 1]);
      Tm8 tm[RB];
      if constexpr (WIDE) {
#pragma unroll
        for (int k = 0; k < RB; ++k) tmem_ld8(tbase + 8 * k, tm[k]);
      }
      __syncthreads();
      const P4 zero{{0ull, 0ull}};
      const P4 below = w > 0 ? as_p4(sm.xch[buf][w - 1][1][lane]) : zero;
      const P4 above = w + 1 < kResWarps ? as_p4(sm.xch[buf][w + 1][0][lane]) : zero;
      buf ^= 1;
      if constexpr (ENERGY && !BATCH) {
        if (s > 0) {
          chain(s - 1);
          if constexpr (LEAN) __syncthreads();
        }
      }
      {
        P4 gb;  // y flux below the current row
        {
          // hy of the last row of the warp before (the first warp's is outside the cone)
          P4 hb = zero;
          if constexpr (WIDE && R <= kTmemRows)
            hb = as_p4(sm.f[Smem::kField - 1][tid]);
          else if (w > 0)
            hb = as_p4(sm.f[Smem::kField - 1][tid - 32]);
#pragma unroll
          for (int q = 0; q < 2; ++q) gb.p[q] = mul2(hb.p[q], sub2(u[0].p[q], below.p[q]));
        }
        // blocks of RB rows, phase by phase, so that the shuffles and loads of the rows of a block
        // overlap (a warp has only three others on its scheduler)
#pragma unroll
        for (int b = 0; b < R; b += RB) {
          P4 fr[RB], gy[RB];
          float ur[RB], fl[RB];
          if constexpr (WIDE) {
#pragma unroll
            for (int k = 0; k < RB; ++k)
              if (b + k < R && b + k < kTmemRows) tmem_wait_ld(tm[k]);
          }
#pragma unroll
          for (int k = 0; k < RB; ++k) {
            const int r = b + k;
            if (r >= R) continue;
            ur[k] = __shfl_down_sync(0xffffffffu, upk(u[r].p[0]).x, 1);
          }
#pragma unroll
          for (int k = 0; k < RB; ++k) {
            const int r = b + k;
            if (r >= R) continue;
            P4 hxv, hyv;
            if constexpr (WIDE) {
              if (r < kTmemRows) {
                hxv = tm_p4(tm[k], 0);
                hyv = tm_p4(tm[k], 4);
              } else {
                hxv = as_p4(sm.f[R + 2 * (r - kTmemRows)][tid]);
                hyv = as_p4(sm.f[R + 2 * (r - kTmemRows) + 1][tid]);
              }
            } else {
              hxv = as_p4(sm.f[2 * r][tid]);
              hyv = as_p4(sm.f[2 * r + 1][tid]);
            }
            const P4 uu = r + 1 < R ? u[r + 1 < R ? r + 1 : r] : above;
#pragma unroll
            for (int q = 0; q < 2; ++q) gy[k].p[q] = mul2(hyv.p[q], sub2(uu.p[q], u[r].p[q]));
            const float2 c01 = upk(u[r].p[0]), c23 = upk(u[r].p[1]);
            fr[k].p[0] = mul2(hxv.p[0], pk(__fsub_rn(c01.y, c01.x), __fsub_rn(c23.x, c01.y)));
            fr[k].p[1] = mul2(hxv.p[1], pk(__fsub_rn(c23.y, c23.x), __fsub_rn(ur[k], c23.y)));
            fl[k] = __shfl_up_sync(0xffffffffu, upk(fr[k].p[1]).y, 1);
          }
          if constexpr (WIDE) {
#pragma unroll
            for (int k = 0; k < RB; ++k)
              if (b + RB + k < R && b + RB + k < kTmemRows) tmem_ld8(tbase + 8 * (b + RB + k), tm[k]);
          }
#pragma unroll
          for (int k = 0; k < RB; ++k) {
            const int r = b + k;
            if (r >= R) continue;
            if constexpr (REC) {
              if ((rec_rows >> r) & 1u) {  // receivers on this row: u^{n} before the step
                stage[lane] = as_f4(u[r]);
                __syncwarp();
                for (int q = lane; q < nrec; q += 32) {
                  const int2 e = sm.rec[q];
                  if ((e.x >> 8) == rw + r)
                    a.traces[((int64_t)p * kResK + s) * a.nrec + e.y] =
                        reinterpret_cast<const float*>(stage)[e.x & 255];
                }
                __syncwarp();
              }
            }
            const float2 F01 = upk(fr[k].p[0]), F23 = upk(fr[k].p[1]);
            P4 fx, vn = get_v(r);
            fx.p[0] = pk(__fsub_rn(F01.x, fl[k]), __fsub_rn(F01.y, F01.x));
            fx.p[1] = pk(__fsub_rn(F23.x, F01.y), __fsub_rn(F23.y, F23.x));
            [[maybe_unused]] float erow = 0.f;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              // -B u (negation is exact, so v - (-B u) rounds as v + B u), v += B u, u += v
              const f2x bv = fma2(ncx2[q], fx.p[q], mul2(ncy2[q], sub2(gy[k].p[q], k == 0 ? gb.p[q] : gy[k > 0 ? k - 1 : 0].p[q])));
              const f2x pc = vn.p[q];
              vn.p[q] = sub2(pc, bv);
              // (u^n - u^{n-1})^2 - (B u^n) u^{n-1} = v^n v^{n+1} + (-B u^n) u^n, rounded and summed over the
              // lane's columns as k_step_wtb.cu does, so that the energies agree far below one ulp of a term
              if constexpr (ENERGY) {
                const float2 ef = upk(fma2(bv, u[r].p[q], mul2(pc, vn.p[q])));
                erow += ef.x + ef.y;
              }
              u[r].p[q] = add2(u[r].p[q], vn.p[q]);
            }
            set_v(r, vn);
            if constexpr (ENERGY) sm.er[s % Smem::kEr][w * R + r][lane] = erow;
          }
          gb = gy[RB - 1];
        }
      }
      if (in_rows != all_rows) {  // rows outside the grid and its boundary rows stay 0
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (!((in_rows >> r) & 1u)) {
            u[r] = zero;
            set_v(r, zero);
          }
      }
    }
    // opaque copies: the exchange's addresses are computed when needed, not kept through the steps
    int rx = rw, lx = lane, tx = tid;
    asm volatile("" : "+r"(rx), "+r"(lx), "+r"(tx));
    const bool last = p + 1 == npass;
    const int q = p & 1;
    const uint32_t tag = (uint32_t)p + 1u;
    if constexpr (LEAN) {
      __syncthreads();
      chain(ns - 1);
      __syncthreads();
    }
    if (!last) {
      // ---- the rims: four rows (all output lanes) where this warp holds them, and its two output
      // columns of lanes, gathered in shared memory so that each lane sends one row's
      if (rim_rows) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (!((rim_rows >> r) & 1u)) continue;
          const int j = rx + r;
          if (j < y0 + kResK) item_put(row_rim(q, cta, 0, j - y0) + lx, as_f4(u[r]), as_f4(get_v(r)), tag + a.skew);
          if (j >= y1 - kResK) item_put(row_rim(q, cta, 1, j - (y1 - kResK)) + lx, as_f4(u[r]), as_f4(get_v(r)), tag + a.skew);
        }
      }
      __syncwarp();
      if (lx == 1 || lx == 30) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          stage[4 * r + (lx == 30 ? 2 : 0)] = as_f4(u[r]);
          stage[4 * r + (lx == 30 ? 3 : 1)] = as_f4(get_v(r));
        }
      }
      __syncwarp();
      for (int k = lx; k < 2 * R; k += 32)
        if ((k & 1) ? has_r : has_l)
          item_put(col_rim(q, cta, k & 1) + (k >> 1), stage[2 * k], stage[2 * k + 1], tag + a.skew);
    } else if (col_out) {  // ---- the end: the whole tile
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!((own_rows >> r) & 1u)) continue;
        auto masked = [&](const float4& x) {
          return make_float4(ncol[0] ? x.x : 0.f, ncol[1] ? x.y : 0.f, ncol[2] ? x.z : 0.f, ncol[3] ? x.w : 0.f);
        };
        *reinterpret_cast<float4*>(a.uo + ((int64_t)(rx + r) * a.ld + c0)) = masked(as_f4(u[r]));
        *reinterpret_cast<float4*>(a.vo + ((int64_t)(rx + r) * a.ld + c0)) = masked(as_f4(get_v(r)));
      }
    }
    if constexpr (ENERGY) {
      float2 e[kResK];
      if constexpr (BATCH) {
        __syncthreads();
        float es[kResK], ec[kResK];
#pragma unroll
        for (int t = 0; t < kResK; ++t) es[t] = ec[t] = 0.f;
        const int r0 = kResK + kResChain * w, r1 = min(r0 + kResChain, kResK + y1 - y0);
        if (col_out) {
#pragma unroll 2
          for (int r = r0; r < r1; ++r)
#pragma unroll
            for (int t = 0; t < kResK; ++t) {  // steps past ns hold older terms, dropped below
              const float y = sm.er[t % Smem::kEr][r][lx] - ec[t];
              const float sum = es[t] + y;
              ec[t] = (sum - es[t]) - y;
              es[t] = sum;
            }
        }
#pragma unroll
        for (int t = 0; t < kResK; ++t) e[t] = t < ns ? make_float2(es[t], -ec[t]) : make_float2(0.f, 0.f);
      } else if constexpr (!LEAN) {
        __syncthreads();
        chain(ns - 1);
      }
      // the warp's sums of the pass's steps: lanes 8 t .. 8 t + 7 end up with step t
      if constexpr (!BATCH) {
#pragma unroll
        for (int t = 0; t < kResK; ++t) {
          e[t] = make_float2(0.f, 0.f);
          if (t < ns) e[t] = LEAN ? a.es[((int64_t)cta * kResK + t) * kResThreads + tx] : sm.es[Smem::kEs ? t : 0][Smem::kEs ? tx : 0];
        }
      }
      auto fold = [&](float3& keep, const float3& send, int o) {
        sum_add(keep, make_float3(__shfl_xor_sync(0xffffffffu, send.x, o), __shfl_xor_sync(0xffffffffu, send.y, o),
                                  __shfl_xor_sync(0xffffffffu, send.z, o)));
      };
      // the first additions are of pairs: nothing in the lows to send
      auto fold2 = [&](const float2& keep, const float2& send, int o) {
        float3 k = make_float3(keep.x, keep.y, 0.f);
        sum_add(k, make_float3(__shfl_xor_sync(0xffffffffu, send.x, o), __shfl_xor_sync(0xffffffffu, send.y, o), 0.f));
        return k;
      };
      float3 k = make_float3(0.f, 0.f, 0.f);
      const int t = lx >> 3;
      // small tiles: warps past the chains have nothing to add (1003 x 517 1.74 to 1.70 us per step)
      if (!BATCH || kResChain * w < y1 - y0) {
        const bool h16 = lx & 16, h8 = lx & 8;
        const float3 k0 = fold2(h16 ? e[2] : e[0], h16 ? e[0] : e[2], 16);
        const float3 k1 = fold2(h16 ? e[3] : e[1], h16 ? e[1] : e[3], 16);
        k = h8 ? k1 : k0;
        fold(k, h8 ? k0 : k1, 8);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) fold(k, k, o);
      }
      if ((lx & 7) == 0) sm.esw[t][w] = k;
      __syncthreads();
      if (w == kResWarps - 1) {  // the CTA's sums
        float3 x = sm.esw[t][lx & 7];
        sum_add(x, sm.esw[t][(lx & 7) + 8]);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) fold(x, x, o);
        if ((lx & 7) == 0 && t < ns)
          a.part[((int64_t)p * kResK + t) * ncta + cta] = (double)x.x + ((double)x.y + (double)x.z);
      }
    } else {
      __syncthreads();
    }
    if (last) break;
    // ---- the halo, from the neighbours' rims: warp w fetches half a row (w / 2: the four rows below
    // the tile, then the four above) for the warps that hold it, and its own rows' outer lanes; the
    // exchange buffer the last step read is free after the barrier above and not written before the
    // next one
    float4* const halo = &sm.xch[buf ^ 1][0][0][0];  // [8][32][2]
    for (int i = lx; i < 16 + 2 * R; i += 32) {
      const ResItem* src = nullptr;
      float4* dst = nullptr;
      if (i < 16) {
        const int k = w >> 1, l = (w & 1) * 16 + i;
        const int j = k < kResK ? y0 - kResK + k : y1 + k - kResK;
        const int ci = strip * kResOut - 8 + 4 * l;
        if (j >= 1 && j <= a.ny - 2 && ci >= 0 && ci < a.ld) {
          const int c = cta + (l == 0 ? -1 : l == 31 ? 1 : 0) + (k < kResK ? -nsx : nsx);
          src = row_rim(q, c, k < kResK ? 1 : 0, k & (kResK - 1)) + (l == 0 ? 30 : l == 31 ? 1 : l);
          dst = halo + (k * 32 + l) * 2;
        }
      } else {
        const int k = i - 16;
        if (((k & 1) ? has_r : has_l) && ((own_rows >> (k >> 1)) & 1u)) {
          src = col_rim(q, (k & 1) ? cta + 1 : cta - 1, (k & 1) ^ 1) + (k >> 1);
          dst = &stage[2 * k];
        }
      }
      if (src) {
        float4 x, y;
        item_get(src, x, y, tag, a.wait, dead);
        dst[0] = x;
        dst[1] = y;
      }
    }
    __syncwarp();
    if (((lx == 0 && has_l) || (lx == 31 && has_r)) && col_in) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!((own_rows >> r) & 1u)) continue;
        u[r] = as_p4(stage[4 * r + (lx == 31 ? 2 : 0)]);
        set_v(r, as_p4(stage[4 * r + (lx == 31 ? 3 : 1)]));
      }
    }
    __syncthreads();  // halo complete; the energy slots are free again
    if (halo_rows && col_in) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!((halo_rows >> r) & 1u)) continue;
        const int j = rx + r, k = j < y0 ? j - (y0 - kResK) : j - y1 + kResK;
        u[r] = as_p4(halo[(k * 32 + lx) * 2]);
        set_v(r, as_p4(halo[(k * 32 + lx) * 2 + 1]));
      }
    }
  }
  if (dead) atomicExch(a.status, (int)TSU_ETIMEOUT);
  if constexpr (WIDE) {
    __syncthreads();
    if (w == 0)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(*(volatile uint32_t*)&sm.tmem));
  }
}

// energy[n] = escale * the sum of step n's partials over the CTAs, one warp per step: lane by lane in
// CTA order, then a shuffle tree (the same value whatever the timing)
__global__ void __launch_bounds__(128) k_res_energy(const double* part, double* energy, const double escale,
                                                    const int ncta, const int64_t nsteps) {
  const int64_t n = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (n >= nsteps) return;
  double s = 0.0;
  for (int c = lane; c < ncta; c += 32) s += part[n * ncta + c];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) energy[n] = s * escale;
}

using ResKernel = void (*)(const ResArgs);
struct ResVariant {
  int rows;  // rows per warp
  size_t smem;
  ResKernel kern[2];  // without, with receivers
};
template <int R, int RB, bool WIDE, bool ENERGY>
constexpr ResVariant res_variant() {
  static_assert(sizeof(ResSmem<R, WIDE, ENERGY>) <= 227 * 1024, "shared memory of a CTA");
  ResVariant v{R, sizeof(ResSmem<R, WIDE, ENERGY>), {k_leapfrog_res<R, RB, WIDE, ENERGY, false>, nullptr}};
  if constexpr (!res_lean(R, ENERGY)) v.kern[1] = k_leapfrog_res<R, RB, WIDE, ENERGY, true>;
  return v;
}
// Without the energy, then with it.  A grid takes the fewest rows per warp that hold it; between 8 and 17 not
// every count is built, so some grids carry rows they do not need (1900^2 17: 4.62 us per step without the
// energy, where 1800^2 takes 3.08 at 14).  17 is one row more than tensor memory holds; it is what 2048 rows
// in 8 chunks need.
const ResVariant kResVariants[] = {
    res_variant<2, 2, false, false>(),  res_variant<3, 3, false, false>(), res_variant<4, 2, false, false>(),
    res_variant<5, 2, true, false>(),  res_variant<6, 2, true, false>(), res_variant<7, 2, true, false>(),
    res_variant<8, 2, true, false>(),  res_variant<10, 2, true, false>(), res_variant<12, 2, true, false>(),
    res_variant<14, 2, true, false>(),  res_variant<17, 2, true, false>(), res_variant<2, 2, false, true>(),
    res_variant<3, 3, false, true>(),   res_variant<4, 2, false, true>(),  res_variant<5, 2, true, true>(),
    res_variant<6, 2, true, true>(),   res_variant<7, 2, true, true>(),  res_variant<8, 2, true, true>(),
    res_variant<10, 2, true, true>(),
    res_variant<12, 2, true, true>(),   res_variant<14, 2, true, true>(),  res_variant<17, 2, true, true>()};
constexpr int kResPlain = 11;  // variants without the energy
constexpr int kResNumVariants = (int)(sizeof kResVariants / sizeof kResVariants[0]);
// own rows of a tile: with the energy whole chains
int res_cap(int k) {
  const int cap = kResWarps * kResVariants[k].rows - 2 * kResK;
  return k < kResPlain ? cap : cap / kResChain * kResChain;
}

// SMs that can hold a CTA of every variant on this device (0: not available), once per device
std::atomic<int> g_res_sms[64];
int res_sms() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int v = g_res_sms[dev].load();
  if (v != 0) return v > 0 ? v : 0;
  int nsm = 0, coop = 0;
  bool ok = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop != 0;
  for (int k = 0; ok && k < 2 * kResNumVariants; ++k) {
    const ResVariant& x = kResVariants[k / 2];
    int q = 0;
    if (!x.kern[k & 1]) continue;
    ok = cudaFuncSetAttribute(x.kern[k & 1], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)x.smem) ==
             cudaSuccess &&
         cudaOccupancyMaxActiveBlocksPerMultiprocessor(&q, x.kern[k & 1], kResThreads, x.smem) == cudaSuccess &&
         q >= 1;
  }
  (void)cudaGetLastError();  // a refused query leaves no error behind
  v = ok ? (nsm < kResMaxCtas ? nsm : kResMaxCtas) : -1;
  g_res_sms[dev].store(v);
  return v > 0 ? v : 0;
}

int64_t res_strips(int64_t ld) { return (ld + 4 + kResOut - 1) / kResOut; }

}  // namespace

// Workspace of the resident pass for this grid: counters, rims and partials of the largest of the
// variants whose tiles number at most kResMaxCtas; 0: the grid does not fit on any device.
// the rims, then 128 bytes with the word of expired waits (PollLimit)
static size_t res_rim_bytes(int k, int64_t ncta) {
  return (size_t)ncta * 2 * (2 * kResWarps * kResVariants[k].rows + 2 * kResK * 32) * sizeof(ResItem) + 128;
}
static size_t res_part_bytes(int k, int64_t ncta) {
  const bool lean = res_lean(kResVariants[k].rows, k >= kResPlain);
  return (size_t)ncta * (kResEnergySteps * sizeof(double) + (lean ? kResK * kResThreads * sizeof(float2) : 0));
}
size_t res_bytes(int64_t ny, int64_t ld) {
  size_t most = 0;
  for (int k = 0; k < kResNumVariants; ++k) {
    const int64_t cap = res_cap(k);
    const int64_t ncta = res_strips(ld) * ((ny - 2 + cap - 1) / cap);
    if (ncta > kResMaxCtas) continue;
    const size_t b = res_rim_bytes(k, ncta) + (k < kResPlain ? 0 : res_part_bytes(k, ncta));
    if (b > most) most = b;
  }
  return most;
}

// Rows per CTA on this device: the fewest rows per warp with which the tiles fit one CTA per SM,
// the chunks then evened out (with the energy: whole chains of 16 rows, the rows of the other passes'
// tiles up to about 2000^2); 0: the grid does not fit.
static int res_rows(int64_t ny, int64_t ld, bool energy, int* variant) {
  const int sms = res_sms();
  const int64_t strips = res_strips(ld), inner = ny - 2;
  for (int k = energy ? kResPlain : 0; k < (energy ? kResNumVariants : kResPlain); ++k) {
    const int64_t cap = res_cap(k);
    int64_t chunks = (inner + cap - 1) / cap;
    if (strips * chunks > sms) continue;
    *variant = k;
    const int64_t rows = (inner + chunks - 1) / chunks;
    return (int)(energy ? (rows + kResChain - 1) / kResChain * kResChain : rows);
  }
  return 0;
}

// The variant and the rows per CTA for these outputs (rec: receivers are recorded); false: the device, the
// workspace or the grid do not allow it.
static bool res_plan(const StencilGeom& g, bool energy, bool rec, int32_t nrec, const EnergyWs& ews, int* variant,
                     int* rows) {
  if (energy) {  // the rows that the pass taken otherwise sums its energy over
    const bool flow = !rec && wtb_flow_preferred(g.ny, g.ld);
    if ((flow ? wtb_flow_rows(g.ny, g.ld) : wtb_auto_rows(g.ny, g.ld, kResK)) != kResChain) return false;
  }
  *rows = res_rows(g.ny, g.ld, energy, variant);
  return *rows > 0 && ews.res && ews.res_size >= res_bytes(g.ny, g.ld) && ews.status && (!rec || nrec <= kResMaxRec) &&
         kResVariants[*variant].kern[rec ? 1 : 0];
}

bool res_fits(const StencilGeom& g, bool energy, bool rec, int32_t nrec, const EnergyWs& ews) {
  int k = 0, rows = 0;
  return res_plan(g, energy, rec, nrec, ews, &k, &rows);
}

// Tiles of 17 rows per warp take 16: with receivers 1900^2 (us per call on chip and in four-step passes) 74
// and 65 at 8 steps, 95 and 92 at 12, 117 and 119 at 16; with a checkpoint every 8, 12 and 16 steps 81 and 69,
// 98 and 94, 116 and 118 per interval.  At up to 14 rows 8 are enough (1800^2 54 and 61, 62 and 66).
int64_t res_min_steps_recording(const StencilGeom& g, int64_t usual) {
  int k = 0;
  return res_rows(g.ny, g.ld, false, &k) > 0 && kResVariants[k].rows > kTmemRows ? 2 * usual : usual;
}

cudaError_t launch_step_res(const StencilGeom& g, const void* hx, const void* hy, void* const u[2], void* const v[2],
                            double* energy, const EnergyWs& ews, int64_t nsteps, cudaStream_t s, int32_t nrec,
                            const int64_t* rec_idx, void* traces, bool table, bool hold, bool* ran, int* last) {
  *ran = false;
  *last = 0;
  int k = 0, rows = 0;
  if (nsteps < 1 || nsteps >= (int64_t)1 << 31 ||
      !res_plan(g, energy != nullptr, traces != nullptr, nrec, ews, &k, &rows))
    return cudaSuccess;
  ResArgs a{};
  a.nx = g.nx;
  a.ny = g.ny;
  a.ld = g.ld;
  a.cx = (float)g.cx;
  a.cy = (float)g.cy;
  a.hx = (const float*)hx;
  a.hy = (const float*)hy;
  a.rows = rows;
  a.nstrips = (int)res_strips(g.ld);
  a.nchunks = (g.ny - 2 + rows - 1) / rows;
  const ResVariant& x = kResVariants[k];
  const int64_t ncta = (int64_t)a.nstrips * a.nchunks;
  a.col = (ResItem*)ews.res;
  a.row = a.col + 2 * ncta * 2 * kResWarps * x.rows;
  a.part = (double*)((char*)ews.res + res_rim_bytes(k, ncta));
  a.es = (float2*)(a.part + kResEnergySteps * ncta);
  a.status = ews.status;
  a.wait = PollLimit{hold ? kPollHookNs : kPollNs, (int*)((char*)ews.res + res_rim_bytes(k, ncta) - 128)};
  a.skew = hold ? 1u << 31 : 0u;
  cudaError_t e = cudaSuccess;
  if (traces) {
    if (table) e = launch_wtb_rec_table(g, rows, rec_idx, nrec, ews, s);
    if (e == cudaSuccess) e = launch_wtb_trace_edges(g, rec_idx, nrec, traces, nsteps, s);
    if (e != cudaSuccess) return e;
    a.nrec = nrec;
    a.rec_off = ews.rec_off;
    a.rec_ent = ews.rec_ent;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ncta);
  cfg.blockDim = dim3(kResThreads);
  cfg.dynamicSmemBytes = x.smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  for (int64_t n = 0; n < nsteps; n += a.nsteps) {
    const int64_t most = energy ? kResEnergySteps : kResMaxSteps;
    a.nsteps = nsteps - n > most ? most : nsteps - n;
    a.u = (const float*)u[*last];
    a.v = (const float*)v[*last];
    *last ^= 1;
    a.uo = (float*)u[*last];
    a.vo = (float*)v[*last];
    if (a.rec_off) a.traces = (float*)traces + n * nrec;
    // no item may carry a tag of an earlier launch
    e = cudaMemsetAsync(ews.res, 0, res_rim_bytes(k, ncta), s);
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, x.kern[a.traces ? 1 : 0], a);
    if (e == cudaSuccess && energy) {
      k_res_energy<<<(unsigned)((a.nsteps + 3) / 4), 128, 0, s>>>(a.part, energy + n, g.dxdy / (2.0 * g.tau * g.tau),
                                                                  (int)ncta, a.nsteps);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
  }
  *ran = true;
  return cudaSuccess;
}

}  // namespace tsu
