// FP64 leapfrog steps on chip (standard form): every step of a call in one cooperative launch for small
// grids, the fields in the registers of one CTA per SM from the first step to the last
// (arXiv:2005.11931, Sec. 2 eq. (2.1) on the Sec. 3.3 box).
//
// One step per launch (k_step64.cu) spends 4 to 6 us on grids of up to about 300^2, of which the FP64
// pipe works 1 to 2: the rest is the launch, the loads and the sums of the energy.  Here a CTA owns 30
// columns (lanes 1 .. 30, a column per lane; lanes 0 and 31 hold the neighbours' edge columns) and a block
// of rows spread over 8 warps, two per scheduler, so that the busiest scheduler has as few rows as
// possible (201^2: 3).  After each step a CTA sends the edge of its tile, 16 bytes per value that carry
// the number of the step, and polls its neighbours' (no flag, no fence); within the CTA the warps
// exchange their first and last rows through shared memory.
//
// Bound by the FP64 pipe (14.5 operations per node and step on the busiest scheduler's rows) and one
// exchange, about 1.2 us, per step.  Measured (GB300, us per step with the energy / without, before, one
// step per launch, and here): 101^2 6.2 / 4.1 and 1.9 / 1.6, 201^2 6.2 / 6.2 and 2.4 / 1.9, 400^2 10.3 / 8.2
// and 6.4 / 5.2, 740^2 24.7 / 20.5 and 17.6 / 14.5; the registers end at 16 rows per warp (about 750^2).
//
// The arithmetic is that of k_step64.cu operation by operation (the states are the same bits).  With
// the energy each lane keeps the term of its rows for 32 steps; then lane t of a warp adds up the 32
// lanes of step t, which costs one FP64 instruction per warp and step instead of a shuffle tree's five.
#include <atomic>

#include "resident64.cuh"
#include "stencil_common.cuh"

namespace tsu {
namespace {
using namespace dev;

constexpr int kR64MaxRows = 16;           // rows per warp
constexpr int kR64Sum = 32;               // steps whose energy terms are summed together
constexpr int64_t kR64MaxSteps = 16384;   // steps per launch (a fraction of a second: see k_step_res.cu)
constexpr int64_t kR64EnergySteps = 512;  // steps per launch with the energy (partials kept)

struct R64Args {
  int32_t nx, ny;
  int64_t ld;
  double cx, cy;
  const double* hx;
  const double* hy;
  double* u;  // u^n, and u^{n + nsteps} at the end
  double* p;  // u^{n-1}, and u^{n + nsteps - 1} at the end
  int rows, nstrips, nchunks;
  int64_t nsteps;
  double* part;  // [step][CTA] energy partials
  ulonglong2* col;    // [2][CTA][2][kR64Rows] first and last own column
  ulonglong2* row;    // [2][CTA][2][32] first and last own row
  int* status;
  double* traces;
  int32_t nrec;
  const int64_t* rec_idx;
  double* seg;  // or nullptr: u^{n+1+k} into seg + k seg_stride, and u, p left as they are
  int64_t seg_stride;
  PollLimit wait;
  uint32_t skew;  // added to the tags sent: 0 (test hook: a number that no reader waits for)
};

struct R64Smem {
  double xch[2][kR64Warps][2][32];  // first and last row of every warp, double buffered
  double es[kR64Sum][kR64Threads + 1];
  double ew[kR64Warps][kR64Sum];
  double stage[kR64Warps][32];
  int2 rec[kResMaxRec];  // (row << 8 | lane, receiver)
  int nrec;
};

template <int R, bool ENERGY>
__global__ void __launch_bounds__(kR64Threads, 1) k_leapfrog_res64(const R64Args a) {
  extern __shared__ __align__(16) unsigned char r64_raw[];
  R64Smem& sm = *reinterpret_cast<R64Smem*>(r64_raw);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int cta = blockIdx.x, ncta = gridDim.x, nsx = a.nstrips;
  const int chunk = cta / nsx, strip = cta - chunk * nsx;
  const int c = strip * kR64Out + lane;
  const int y0 = 1 + chunk * a.rows, y1 = min(y0 + a.rows, a.ny - 1), rows = y1 - y0;
  // the first rows % 8 warps take one row more: schedulers (w % 4) stay within one row of each other
  const int base = rows / kR64Warps, extra = rows - base * kR64Warps;
  const int cnt = base + (w < extra ? 1 : 0), r0 = w * base + min(w, extra), j0 = y0 + r0;
  const int wl = min(rows, kR64Warps) - 1;  // the last warp with rows
  const bool in = c < a.nx;
  const bool node = lane >= 1 && lane <= 30 && c <= a.nx - 2;
  const bool has_l = strip > 0, has_r = strip + 1 < nsx, has_d = chunk > 0, has_u = chunk + 1 < a.nchunks;
  auto at = [&](const double* f, int j) { return in ? __ldcg(f + (int64_t)j * a.ld + c) : 0.0; };

  double u[R], p[R], hx[R], hy[R], hd = 0.0, below = 0.0, above = 0.0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    u[r] = p[r] = hx[r] = hy[r] = 0.0;
    if (r < cnt) {
      u[r] = at(a.u, j0 + r);
      p[r] = node ? at(a.p, j0 + r) : 0.0;
      hx[r] = at(a.hx, j0 + r);
      hy[r] = at(a.hy, j0 + r);
    }
  }
  if (cnt > 0) {
    hd = at(a.hy, j0 - 1);
    below = at(a.u, j0 - 1);
    above = at(a.u, j0 + cnt);
  }
  // receivers of the tile's own nodes; those on the boundary or outside the grid record 0
  uint32_t rec_rows = 0;
  int nrec = 0;
  if (a.traces) {
    if (tid == 0) sm.nrec = 0;
    __syncthreads();
    for (int q = tid; q < a.nrec; q += kR64Threads) {
      const int64_t v = a.rec_idx[q];
      const int64_t j = v >= 0 && v < (int64_t)a.ny * a.ld ? v / a.ld : 0, i = v - j * a.ld;
      if (j >= 1 && j <= a.ny - 2 && i >= 1 && i <= a.nx - 2) {
        if (j >= y0 && j < y1 && (i - 1) / kR64Out == strip)
          sm.rec[atomicAdd(&sm.nrec, 1)] = make_int2((int)(j << 8) | (int)(i - strip * kR64Out), q);
      } else if (cta == 0) {
        for (int64_t n = 0; n < a.nsteps; ++n) a.traces[n * a.nrec + q] = 0.0;
      }
    }
    __syncthreads();
    nrec = sm.nrec;
    for (int q = 0; q < nrec; ++q) {
      const int r = (sm.rec[q].x >> 8) - j0;
      if (r >= 0 && r < cnt) rec_rows |= 1u << r;
    }
  }
  auto col_rim = [&](int q, int k, int side) { return a.col + (((int64_t)q * ncta + k) * 2 + side) * kR64Rows + r0; };
  auto row_rim = [&](int q, int k, int side) { return a.row + (((int64_t)q * ncta + k) * 2 + side) * 32 + lane; };
  bool dead = false;
  const double cx = a.cx, cy = a.cy;

  for (int n = 0; n < (int)a.nsteps; ++n) {
    if (rec_rows) {  // u^n at the receivers
#pragma unroll
      for (int r = 0; r < R; ++r)
        if ((rec_rows >> r) & 1u) {
          sm.stage[w][lane] = u[r];
          __syncwarp();
          for (int q = lane; q < nrec; q += 32)
            if ((sm.rec[q].x >> 8) == j0 + r)
              a.traces[(int64_t)n * a.nrec + sm.rec[q].y] = sm.stage[w][sm.rec[q].x & 255];
          __syncwarp();
        }
    }
    double e = 0.0, gd = 0.0;
    if (cnt > 0) gd = __dmul_rn(hd, __dsub_rn(u[0], below));
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (r >= cnt) break;
      const double uc = u[r], un = r + 1 < R ? (r + 1 < cnt ? u[r + 1 < R ? r + 1 : r] : above) : above;
      const double ur = __shfl_down_sync(0xffffffffu, uc, 1);
      const double fr = __dmul_rn(hx[r], __dsub_rn(ur, uc));
      const double fl = __shfl_up_sync(0xffffffffu, fr, 1);
      const double gu = __dmul_rn(hy[r], __dsub_rn(un, uc));
      const double b = __fma_rn(cx, __dsub_rn(fr, fl), __dmul_rn(cy, __dsub_rn(gu, gd)));
      if constexpr (ENERGY) {
        // (u^n - u^{n-1})^2 - (B u^n) u^{n-1}
        const double d = __dsub_rn(uc, p[r]);
        e = __fma_rn(-b, p[r], r == 0 ? __dmul_rn(d, d) : __fma_rn(d, d, e));
      }
      const double unew = __dadd_rn(__fma_rn(2.0, uc, -p[r]), b);
      p[r] = uc;
      u[r] = node ? unew : 0.0;
      gd = gu;
    }
    if constexpr (ENERGY) sm.es[n & (kR64Sum - 1)][tid] = node ? e : 0.0;
    if (a.seg && node) {
      double* d = a.seg + (int64_t)n * a.seg_stride + (int64_t)j0 * a.ld + c;
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (r < cnt) d[(int64_t)r * a.ld] = u[r];
    }
    const bool last = n + 1 == (int)a.nsteps;
    if (!last) {
      const int q = n & 1;
      const uint32_t tag = (uint32_t)n + 1u;
      // the edges of the tile: own columns 1 and 30 (lanes), first and last row
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (r < cnt && ((lane == 1 && has_l) || (lane == 30 && has_r)))
          put64(col_rim(q, cta, lane == 30 ? 1 : 0) + r, u[r], tag + a.skew);
      double top = u[0];
#pragma unroll
      for (int r = 1; r < R; ++r)
        if (r < cnt) top = u[r];
      if (cnt > 0) {
        if (w == 0 && has_d) put64(row_rim(q, cta, 0), u[0], tag + a.skew);
        if (w == wl && has_u) put64(row_rim(q, cta, 1), top, tag + a.skew);
        sm.xch[q][w][0][lane] = u[0];
        sm.xch[q][w][1][lane] = top;
      }
      __syncthreads();
      if (cnt > 0) {
        // the neighbours' edges: every load issued before the first is waited for
        const bool edge = (lane == 0 && has_l) || (lane == 31 && has_r);
        const ulonglong2* cs = col_rim(q, lane == 0 ? cta - 1 : cta + 1, lane == 0 ? 1 : 0);
        ulonglong2 x[R], xd, xu;
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (edge && r < cnt) x[r] = try64(cs + r);
        const bool dn = w == 0 && has_d && node, up = w == wl && has_u && node;
        const ulonglong2 *ds = row_rim(q, cta - nsx, 1), *us = row_rim(q, cta + nsx, 0);
        if (dn) xd = try64(ds);
        if (up) xu = try64(us);
        if (w > 0) below = sm.xch[q][w - 1][1][lane];
        if (w < wl) above = sm.xch[q][w + 1][0][lane];
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (edge && r < cnt) u[r] = get64(x[r], cs + r, tag, a.wait, dead);
        if (dn) below = get64(xd, ds, tag, a.wait, dead);
        if (up) above = get64(xu, us, tag, a.wait, dead);
        __syncwarp();
      }
    }
    if constexpr (ENERGY) {
      if ((n & (kR64Sum - 1)) == kR64Sum - 1 || last) {
        __syncthreads();
        const int m = n & (kR64Sum - 1);  // steps n - m .. n wait
        double s[4] = {0.0, 0.0, 0.0, 0.0};
        if (lane <= m) {
#pragma unroll
          for (int k = 0; k < 32; ++k) s[k & 3] += sm.es[lane][w * 32 + k];
        }
        sm.ew[w][lane] = (s[0] + s[1]) + (s[2] + s[3]);
        __syncthreads();
        if (w == 0 && lane <= m) {
          double t = 0.0;
          for (int k = 0; k < kR64Warps; ++k) t += sm.ew[k][lane];
          a.part[(int64_t)(n - m + lane) * ncta + cta] = t;
        }
      }
    }
  }
  if (node && !a.seg) {
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (r < cnt) {
        a.u[(int64_t)(j0 + r) * a.ld + c] = u[r];
        a.p[(int64_t)(j0 + r) * a.ld + c] = p[r];
      }
  }
  if (dead && a.status) atomicExch(a.status, (int)TSU_ETIMEOUT);
}

using R64Kernel = void (*)(const R64Args);
struct R64Variant {
  int rows;
  R64Kernel kern[2];  // without, with the energy
};
template <int R>
constexpr R64Variant r64_variant() {
  return R64Variant{R, {k_leapfrog_res64<R, false>, k_leapfrog_res64<R, true>}};
}
const R64Variant kR64Variants[] = {r64_variant<1>(), r64_variant<2>(), r64_variant<3>(),
                                   r64_variant<4>(), r64_variant<6>(), r64_variant<8>(),
                                   r64_variant<12>(), r64_variant<kR64MaxRows>()};
constexpr int kR64Num = (int)(sizeof kR64Variants / sizeof kR64Variants[0]);

// SMs that hold a CTA of every variant on this device (0: not available), once per device
std::atomic<int> g_r64_sms[64];
int r64_sms() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int v = g_r64_sms[dev].load();
  if (v != 0) return v > 0 ? v : 0;
  int nsm = 0, coop = 0;
  bool ok = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop != 0;
  for (int k = 0; ok && k < 2 * kR64Num; ++k) {
    const R64Kernel kern = kR64Variants[k / 2].kern[k & 1];
    int q = 0;
    ok = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(R64Smem)) ==
             cudaSuccess &&
         cudaOccupancyMaxActiveBlocksPerMultiprocessor(&q, kern, kR64Threads, sizeof(R64Smem)) == cudaSuccess &&
         q >= 1;
  }
  (void)cudaGetLastError();  // a refused query leaves no error behind
  v = ok ? (nsm < kResMaxCtas ? nsm : kResMaxCtas) : -1;
  g_r64_sms[dev].store(v);
  return v > 0 ? v : 0;
}

static_assert(kR64Warps * kR64MaxRows <= kR64Rows, "rows of a rim");

}  // namespace

// Workspace for grids of this many rows of ld elements; 0: none of them fits.
size_t res64_bytes(int64_t ny, int64_t ld) {
  const int64_t least = r64_strips(ld - 31) * ((ny - 2 + kR64Rows - 1) / kR64Rows);  // nx > ld - 32 usually
  return least <= kResMaxCtas ? kR64RimBytes + (size_t)kR64EnergySteps * kResMaxCtas * sizeof(double) : 0;
}

// The variant and the rows per CTA (one CTA per SM, as many as fit); -1: the grid does not fit.
static int r64_plan(const StencilGeom& g, int64_t* rows) {
  const int64_t sms = r64_sms(), strips = r64_strips(g.nx), inner = g.ny - 2;
  if (sms <= 0 || strips < 1 || strips > sms || g.ny >= 1 << 22) return -1;
  *rows = (inner + sms / strips - 1) / (sms / strips);
  const int64_t per_warp = (*rows + kR64Warps - 1) / kR64Warps;
  for (int k = 0; k < kR64Num; ++k)
    if (kR64Variants[k].rows >= per_warp) return k;
  return -1;
}
static bool r64_workspace(const EnergyWs& ews) {
  return ews.res && ews.status &&
         ews.res_size >= kR64RimBytes + (size_t)kR64EnergySteps * kResMaxCtas * sizeof(double);
}
bool res64_fits(const StencilGeom& g, const EnergyWs& ews) {
  int64_t rows = 0;
  return r64_workspace(ews) && r64_plan(g, &rows) >= 0;
}

static R64Args r64_args(const StencilGeom& g, const void* hx, const void* hy, const void* u, const void* p, int64_t rows,
                        void* rims, bool hold) {
  R64Args a{};
  a.wait = r64_limit(rims, hold);
  a.skew = hold ? 1u << 31 : 0u;
  a.nx = g.nx;
  a.ny = g.ny;
  a.ld = g.ld;
  a.cx = g.cx;
  a.cy = g.cy;
  a.hx = (const double*)hx;
  a.hy = (const double*)hy;
  a.u = (double*)u;
  a.p = (double*)p;
  a.rows = (int)rows;
  a.nstrips = (int)r64_strips(g.nx);
  a.nchunks = (int)((g.ny - 2 + rows - 1) / rows);
  a.col = (ulonglong2*)rims;
  a.row = a.col + (int64_t)2 * a.nstrips * a.nchunks * 2 * kR64Rows;
  return a;
}

static cudaError_t r64_launch(const R64Args& a, R64Kernel kern, cudaStream_t s) {
  // no value may carry a tag of an earlier launch
  const cudaError_t e = cudaMemsetAsync(a.col, 0, kR64RimBytes, s);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.nstrips * a.nchunks));
  cfg.blockDim = dim3(kR64Threads);
  cfg.dynamicSmemBytes = sizeof(R64Smem);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

cudaError_t launch_step_res64(const StencilGeom& g, const void* hx, const void* hy, void* u, void* p, double* energy,
                              const EnergyWs& ews, int64_t nsteps, cudaStream_t s, int32_t nrec,
                              const int64_t* rec_idx, void* traces, bool hold, bool* ran) {
  *ran = false;
  int64_t rows = 0;
  const int k = r64_workspace(ews) ? r64_plan(g, &rows) : -1;
  if (k < 0 || nsteps >= 1ll << 31 || (traces && nrec > kResMaxRec)) return cudaSuccess;
  R64Args a = r64_args(g, hx, hy, u, p, rows, ews.res, hold);
  a.part = (double*)((char*)ews.res + kR64RimBytes);
  a.status = ews.status;
  a.nrec = traces ? nrec : 0;
  a.rec_idx = rec_idx;
  for (int64_t n = 0; n < nsteps; n += a.nsteps) {
    const int64_t most = energy ? kR64EnergySteps : kR64MaxSteps;
    a.nsteps = nsteps - n > most ? most : nsteps - n;
    if (nsteps - n - a.nsteps == 1) a.nsteps -= 1;  // no launch of a single step (it writes in place)
    a.traces = traces ? (double*)traces + n * nrec : nullptr;
    cudaError_t e = r64_launch(a, kR64Variants[k].kern[energy ? 1 : 0], s);
    if (e == cudaSuccess && energy)
      e = launch_energy64(g, a.part, (int64_t)a.nstrips * a.nchunks, a.nsteps, energy + n, s);
    if (e != cudaSuccess) return e;
  }
  *ran = true;
  return cudaSuccess;
}

size_t res64_seg_bytes(const StencilGeom& g) {
  return r64_strips(g.nx) * ((g.ny - 2 + kR64Rows - 1) / kR64Rows) <= kResMaxCtas ? kR64RimBytes : 0;
}

cudaError_t launch_step_res64_seg(const StencilGeom& g, const void* hx, const void* hy, const void* u, const void* p,
                                  void* seg, int64_t seg_stride, int64_t nsteps, void* ws, cudaStream_t s, bool hold,
                                  bool* ran) {
  *ran = false;
  int64_t rows = 0;
  const int k = ws ? r64_plan(g, &rows) : -1;
  if (k < 0 || nsteps < 1 || nsteps > kR64MaxSteps) return cudaSuccess;
  R64Args a = r64_args(g, hx, hy, u, p, rows, ws, hold);
  a.nsteps = nsteps;
  a.seg = (double*)seg;
  a.seg_stride = seg_stride;
  const cudaError_t e = r64_launch(a, kR64Variants[k].kern[0], s);
  *ran = e == cudaSuccess;
  return e;
}

}  // namespace tsu
