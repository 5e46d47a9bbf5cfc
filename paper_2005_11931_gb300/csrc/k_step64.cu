// FP64 leapfrog and reverse steps, one step per launch (arXiv:2005.11931, Sec. 2 eq. (2.1) on the
// Sec. 3.3 box; the schemes of k_step.cu and k_adjoint.cu).
//
// The GB300 issues two FP64 operations per SM and clock (a warp instruction every 64 clocks on each
// of the four schedulers), so these passes are bound by the number of FP64 instructions and by how
// evenly their rows spread over the 608 schedulers; memory waits behind them.  Hence:
//  - every face flux is computed once: the x flux left of a lane comes from the lane on the left, the y
//    flux below a row from the row before (10 FP64 operations per node and step instead of 16, and 14.5
//    with the energy instead of 23; reverse step 17 instead of 28);
//  - a lane holds one column, a warp 32, of which 31 are output (lane 0 only supplies its flux): odd
//    widths waste few lanes (201 columns: 7 strips of 31, against 4 of 64 with 16-byte vectors);
//  - a warp takes a tile of its own, and the rows per tile minimise the rows of the busiest scheduler
//    (step64_rows);
//  - the fields of four rows are loaded before the first of them is used.
// Measured (GB300, us per step, before and after): with the energy 201^2 13.9 and 6.2 (the launch: a step
// takes a multiple of 2.05 us back to back), 2048^2 196 and 127 (the FP64 pipe 84 % active);
// without it 2048^2 114 and 97; a 257^2 gradient of 300 steps 9.5 and 5.2 ms.  Programmatic dependent
// launches were slower (201^2 11.1): the early CTAs doubled up on some SMs.
#include "stencil_common.cuh"

namespace tsu {
namespace {
using namespace dev;

constexpr int kS64Out = kStep64Cols;  // output columns of a strip (lanes 1 .. 31)
constexpr int kS64Warps = 4;   // tiles per CTA, one per scheduler
constexpr int kS64Batch = 4;   // rows loaded together

struct S64Geom {
  int32_t nx, ny;
  int64_t ld;
  double cx, cy;
  int rows, strips, ntiles;
};

// B u at one node from its four face fluxes
__device__ __forceinline__ double b64(const S64Geom& g, double fr, double fl, double gu, double gd) {
  return __fma_rn(g.cx, __dsub_rn(fr, fl), __dmul_rn(g.cy, __dsub_rn(gu, gd)));
}

// Sum of the CTAs' energy partials (at most 2^30), by a CTA of kS64Warps warps; the result is thread 0's.  The
// additions near the top of a tree make the rounding error of the whole sum (those of the many small sums
// below average out), so this one is exact: every partial becomes an integer of 128 bits in units of 2^-92
// times the largest's power of two, and the sum is rounded once.  Relative error of energies against
// binary128, rms over random fields at 101^2, 201^2, 400^2 and 1024^2: 0.8, 0.8, 0.7 and 0.6e-16 (on chip 0.8,
// 0.8, 0.8); with plain FP64 additions here 1.1, 1.1, 1.3 and 1.6e-16 (on chip 1.4, 1.4, 1.5); plain here and every term compensated
// below (3 more FP64 operations per node) 1.0, 1.2, 1.1 and 1.4e-16.  Integers also because an FP64
// instruction takes 64 clocks of a scheduler: keeping the errors in FP64 (two-sum) cost 2 us per sum.
__device__ double partials_sum(const double* part, const int n) {
  __shared__ int top[kS64Warps];
  __shared__ __int128 red[kS64Warps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  auto exponent = [](const double x) { return (int)(__double_as_longlong(x) >> 52) & 0x7ff; };
  int e = 1;
  for (int q = threadIdx.x; q < n; q += kS64Warps * 32) e = max(e, exponent(__ldcg(part + q)));
  e = __reduce_max_sync(0xffffffffu, e);
  if (lane == 0) top[w] = e;
  __syncthreads();
  for (int q = 0; q < kS64Warps; ++q) e = max(e, top[q]);
  if (e == 0x7ff) {  // infinities or NaN
    double s = 0.0;
    if (threadIdx.x == 0)
      for (int q = 0; q < n; ++q) s += __ldcg(part + q);
    return s;
  }
  __int128 sum = 0;
  for (int q = threadIdx.x; q < n; q += kS64Warps * 32) {
    const double x = __ldcg(part + q);
    const long long bits = __double_as_longlong(x);
    const int f = exponent(x), down = e - max(f, 1);  // bits below the largest
    const long long m = (bits & 0xfffffffffffffll) | (f > 0 ? 1ll << 52 : 0);
    const __int128 v = down <= 40 ? (__int128)m << (40 - down) : (__int128)(down - 40 < 64 ? m >> (down - 40) : 0);
    sum += bits < 0 ? -v : v;
  }
  for (int k = 16; k > 0; k >>= 1) {
    const unsigned long long lo = __shfl_down_sync(0xffffffffu, (unsigned long long)sum, k);
    const long long hi = __shfl_down_sync(0xffffffffu, (long long)(sum >> 64), k);
    sum += ((__int128)hi << 64) | lo;
  }
  if (lane == 0) red[w] = sum;
  __syncthreads();
  if (threadIdx.x != 0) return 0.0;
  for (int q = 1; q < kS64Warps; ++q) sum += red[q];
  // the top 64 bits (those below them only decide ties), rounded once
  unsigned __int128 mag = sum < 0 ? (unsigned __int128)-sum : (unsigned __int128)sum;
  const unsigned long long hi = (unsigned long long)(mag >> 64);
  const int drop = hi ? 64 - __clzll((long long)hi) : 0;
  unsigned long long m = (unsigned long long)(mag >> drop);
  if (drop && (mag & (((unsigned __int128)1 << drop) - 1))) m |= 1;
  const double s = ldexp(__ull2double_rn(m), drop + e - 1023 - 52 - 40);
  return sum < 0 ? -s : s;
}

// FORM 0: standard (p = u^{n-1}, out = u^{n+1}, may be written over p); FORM 1: increment (p = v^n updated
// in place, out = u^{n+1}).  MANY: several tiles per warp, where the caller has no room for one energy
// partial per four tiles (the loop costs 0.5 % at 2048^2, so the other launches do without).
template <int FORM, bool STORE, bool ENERGY, bool MANY = false>
__global__ void __launch_bounds__(kS64Warps * 32) k_leapfrog64(const S64Geom g, const double* __restrict__ hx,
                                                               const double* __restrict__ hy,
                                                               const double* u, const double* p_in,
                                                               double* p_out, double* u_next, const PassOut o,
                                                               const double escale) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // receivers: u^n at the receiver nodes, by the first CTA (u is read-only in this pass)
  if (o.trace && blockIdx.x == 0) {
    const int64_t total = (int64_t)g.ny * g.ld;
    for (int r = threadIdx.x; r < o.nrec; r += blockDim.x) {
      const int64_t q = o.rec_idx[r];
      ((double*)o.trace)[r] = (q >= 0 && q < total) ? u[q] : 0.0;  // out-of-range receivers read 0
    }
  }
  double es = 0.0, ec = 0.0;  // compensated energy sum of this lane
  for (int tile = blockIdx.x * kS64Warps + w; tile < g.ntiles; tile += gridDim.x * kS64Warps) {
    const int chunk = tile / g.strips, strip = tile - chunk * g.strips;
    const int c = strip * kS64Out + lane - 1;
    const int j0 = 1 + chunk * g.rows, j1 = min(j0 + g.rows, g.ny - 1);
    const bool in = c >= 0 && c < g.nx;
    double fx[kS64Batch], fy[kS64Batch], hd = 0.0;
    auto faces = [&](int jb) {
#pragma unroll
      for (int k = 0; k < kS64Batch; ++k) {
        const int64_t q = (int64_t)(jb + k) * g.ld + c;
        const bool ok = in && jb + k < j1;
        fx[k] = ok ? __ldg(hx + q) : 0.0;
        fy[k] = ok ? __ldg(hy + q) : 0.0;
      }
    };
    faces(j0);
    if (in) hd = __ldg(hy + (int64_t)(j0 - 1) * g.ld + c);
    const bool out = lane >= 1 && c <= g.nx - 2;  // the strips cover columns 0 .. nx - 2
    const bool node = out && c >= 1;
    const bool tail = lane == 31 && c + 1 < g.nx;
    double uc = in ? __ldcg(u + (int64_t)j0 * g.ld + c) : 0.0;
    double gd = __dmul_rn(hd, __dsub_rn(uc, in ? __ldcg(u + (int64_t)(j0 - 1) * g.ld + c) : 0.0));
    for (int jb = j0; jb < j1; jb += kS64Batch) {
      double un[kS64Batch], pv[kS64Batch], ux[kS64Batch];
      if (jb > j0) faces(jb);
#pragma unroll
      for (int k = 0; k < kS64Batch; ++k) {
        const int j = jb + k;
        const int64_t q = (int64_t)j * g.ld + c;
        const bool ok = in && j < j1;
        un[k] = ok ? __ldcg(u + q + g.ld) : 0.0;
        pv[k] = ok && out ? __ldcg(p_in + q) : 0.0;
        ux[k] = tail && j < j1 ? __ldcg(u + q + 1) : 0.0;
      }
      double e = 0.0;
#pragma unroll
      for (int k = 0; k < kS64Batch; ++k) {
        const int j = jb + k;
        if (j >= j1) break;
        double ur = __shfl_down_sync(0xffffffffu, uc, 1);
        if (lane == 31) ur = ux[k];
        const double fr = __dmul_rn(fx[k], __dsub_rn(ur, uc));
        const double fl = __shfl_up_sync(0xffffffffu, fr, 1);
        const double gu = __dmul_rn(fy[k], __dsub_rn(un[k], uc));
        const double b = b64(g, fr, fl, gu, gd);
        const int64_t q = (int64_t)j * g.ld + c;
        double unew, vnew = 0.0, d;
        if constexpr (FORM == 0) {
          unew = __dadd_rn(__fma_rn(2.0, uc, -pv[k]), b);  // 2 u is exact
        } else {
          vnew = __dadd_rn(pv[k], b);
          unew = __dadd_rn(uc, vnew);
        }
        if constexpr (ENERGY) {
          // (u^n - u^{n-1})^2 - (B u^n) u^{n-1}
          const double up = FORM == 0 ? pv[k] : __dsub_rn(uc, pv[k]);
          d = FORM == 0 ? __dsub_rn(uc, up) : pv[k];
          const double t = __fma_rn(-b, up, k == 0 ? __dmul_rn(d, d) : __fma_rn(d, d, e));
          e = node ? t : 0.0;
        }
        if (o.ckpt_a && out) {  // checkpoint copy of the state read by this pass
          ((double*)o.ckpt_a)[q] = FORM == 0 ? pv[k] : uc;
          ((double*)o.ckpt_b)[q] = FORM == 0 ? uc : pv[k];
        }
        if (STORE && out) {
          u_next[q] = node ? unew : 0.0;
          if constexpr (FORM == 1) p_out[q] = node ? vnew : 0.0;
        }
        uc = un[k];
        gd = gu;
      }
      if constexpr (ENERGY) {
        const double y = __dsub_rn(e, ec), s = __dadd_rn(es, y);
        ec = __dsub_rn(__dsub_rn(s, es), y);
        es = s;
      }
    }
    // a checkpoint slot holds zeros on the boundary and in the padding
    if (o.ckpt_a) {
      if (strip == g.strips - 1)
        for (int j = j0; j < j1; ++j)
          for (int64_t i = g.nx - 1 + lane; i < g.ld; i += 32) {
            ((double*)o.ckpt_a)[(int64_t)j * g.ld + i] = 0.0;
            ((double*)o.ckpt_b)[(int64_t)j * g.ld + i] = 0.0;
          }
      if (strip == 0) {
        for (int64_t i = lane; i < g.ld; i += 32) {
          if (j0 == 1) ((double*)o.ckpt_a)[i] = ((double*)o.ckpt_b)[i] = 0.0;
          if (j1 == g.ny - 1)
            ((double*)o.ckpt_a)[(int64_t)(g.ny - 1) * g.ld + i] = ((double*)o.ckpt_b)[(int64_t)(g.ny - 1) * g.ld + i] =
                0.0;
        }
      }
    }
    if constexpr (!MANY) break;
  }
  if constexpr (ENERGY) {
    __shared__ double red[kS64Warps];
    __shared__ bool last;
    double v = __dsub_rn(es, ec);
    for (int s = 16; s > 0; s >>= 1) v += __shfl_down_sync(0xffffffffu, v, s);
    if (lane == 0) red[w] = v;
    __syncthreads();
    double* part = o.defer ? o.defer : o.ews.partials;
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int q = 0; q < kS64Warps; ++q) s += red[q];
      part[blockIdx.x] = s;
    }
    if (o.defer) return;  // summed after several steps by k_energy64
    if (threadIdx.x == 0) {
      __threadfence();
      last = atomicAdd(o.ews.counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const double t = partials_sum(part, (int)gridDim.x);
    if (threadIdx.x == 0) {
      *o.energy = t * escale;
      *o.ews.counter = 0u;
    }
  }
}

// energy[n] of the steps whose partials wait in part[n][ncta], one CTA per step, in the order of the
// reduction above
__global__ void __launch_bounds__(kS64Warps * 32) k_energy64(const double* part, double* energy, const double escale,
                                                             const int ncta) {
  const double t = partials_sum(part + (int64_t)blockIdx.x * ncta, ncta);
  if (threadIdx.x == 0) energy[blockIdx.x] = t * escale;
}

// lam^n = (2 lam^{n+1} - lam^{n+2}) + B lam^{n+1} over lam^{n+2}, and both face gradients += those of this
// step, from lam^{n+1} and u^n (k_adjoint.cu, kAdjStep)
__global__ void __launch_bounds__(kS64Warps * 32) k_adjoint64(const S64Geom g, const double* __restrict__ hx,
                                                              const double* __restrict__ hy,
                                                              const double* lam, double* lam_pp, const double* u, double* gx,
                                                              double* gy, const RecBuckets rb) {
  const int lane = threadIdx.x & 31;
  const int tile = blockIdx.x * kS64Warps + (threadIdx.x >> 5);
  if (tile >= g.ntiles) return;
  const int chunk = tile / g.strips, strip = tile - chunk * g.strips;
  const int c = strip * kS64Out + lane - 1;
  const bool in = c >= 0 && c < g.nx;
  const bool out = lane >= 1 && c <= g.nx - 2;
  const bool node = out && c >= 1;
  const bool tail = lane == 31 && c + 1 < g.nx;
  const double gwx = -g.cx, gwy = -g.cy;
  const int j0 = 1 + chunk * g.rows, j1 = min(j0 + g.rows, g.ny - 1);
  // u^n with its boundary nodes read as zero
  const bool unode = c >= 1 && c <= g.nx - 2, utail = lane == 31 && c + 1 <= g.nx - 2;
  auto at = [&](const double* f, int j) { return in ? __ldcg(f + (int64_t)j * g.ld + c) : 0.0; };
  double lc = at(lam, j0);
  double uc = unode ? __ldcg(u + (int64_t)j0 * g.ld + c) : 0.0;
  double gd = __dmul_rn(at(hy, j0 - 1), __dsub_rn(lc, at(lam, j0 - 1)));
  constexpr int kB = 2;
  for (int jb = j0; jb < j1; jb += kB) {
    double ln[kB], lp[kB], un[kB], fx[kB], fy[kB], lx[kB], ux[kB], ax[kB], ay[kB];
#pragma unroll
    for (int k = 0; k < kB; ++k) {
      const int j = jb + k;
      const int64_t q = (int64_t)j * g.ld + c;
      const bool ok = in && j < j1;
      ln[k] = ok ? __ldcg(lam + q + g.ld) : 0.0;
      lp[k] = ok && out ? __ldcg(lam_pp + q) : 0.0;
      fx[k] = ok ? __ldg(hx + q) : 0.0;
      fy[k] = ok ? __ldg(hy + q) : 0.0;
      un[k] = unode && j < j1 && j + 1 <= g.ny - 2 ? __ldcg(u + q + g.ld) : 0.0;
      lx[k] = tail && j < j1 ? __ldcg(lam + q + 1) : 0.0;
      ux[k] = utail && j < j1 ? __ldcg(u + q + 1) : 0.0;
      ax[k] = ok && out ? __ldcg(gx + q) : 0.0;
      ay[k] = ok && out ? __ldcg(gy + q) : 0.0;
    }
#pragma unroll
    for (int k = 0; k < kB; ++k) {
      const int j = jb + k;
      if (j >= j1) break;
      double lr = __shfl_down_sync(0xffffffffu, lc, 1), ur = __shfl_down_sync(0xffffffffu, uc, 1);
      if (lane == 31) {
        lr = lx[k];
        ur = ux[k];
      }
      const double dlx = __dsub_rn(lr, lc), dly = __dsub_rn(ln[k], lc);
      const double fr = __dmul_rn(fx[k], dlx), gu = __dmul_rn(fy[k], dly);
      const double fl = __shfl_up_sync(0xffffffffu, fr, 1);
      const double b = b64(g, fr, fl, gu, gd);
      const double val = __dadd_rn(__fma_rn(2.0, lc, -lp[k]), b);
      // x-face (i, i+1) on this row, y-face (j, j+1) on this column (interior columns)
      const double px = __dmul_rn(dlx, __dsub_rn(ur, uc)), py = __dmul_rn(dly, __dsub_rn(un[k], uc));
      if (out) {
        const int64_t q = (int64_t)j * g.ld + c;
        lam_pp[q] = node ? val : 0.0;
        gx[q] = __fma_rn(gwx, px, ax[k]);
        if (node) gy[q] = __fma_rn(gwy, py, ay[k]);
        // y-face (0, 1), where both fields are 0 below
        if (j == 1 && node) gy[c] = __fma_rn(gwy, __dmul_rn(lc, uc), __ldcg(gy + c));
      }
      lc = ln[k];
      uc = un[k];
      gd = gu;
    }
  }
  // receiver injection lam^n += g^n at this tile's receivers, in receiver order
  if (rb.off) {
    __syncwarp();
    if (lane == 0)
      for (int q = rb.off[tile]; q < rb.off[tile + 1]; ++q) {
        const int r = rb.ord[q];
        double* d = lam_pp + rb.idx[r];
        *d += ((const double*)rb.g)[r];
      }
  }
}

S64Geom s64_geom(const StencilGeom& g, int rows) {
  S64Geom s;
  s.nx = g.nx;
  s.ny = g.ny;
  s.ld = g.ld;
  s.cx = g.cx;
  s.cy = g.cy;
  s.rows = rows > 0 ? rows : step64_rows(g.nx, g.ny);
  s.strips = step64_strips(g.nx);
  s.ntiles = s.strips * ((g.ny - 2 + s.rows - 1) / s.rows);
  return s;
}

template <int FORM>
cudaError_t step64(const StencilGeom& g, const void* hx, const void* hy, const void* p, const void* u, void* v,
                   void* u_next, const PassOut& o, bool store, int rows, cudaStream_t s) {
  const S64Geom q = s64_geom(g, rows);
  int64_t grid = (q.ntiles + kS64Warps - 1) / kS64Warps;
  const double scale = g.dxdy / (2.0 * g.tau * g.tau);
  const bool many = o.energy && !o.defer && grid > o.ews.capacity;
  if (many) grid = o.ews.capacity;
  if (grid < 1) return cudaErrorInvalidValue;
  auto run = [&](auto kern) {
    kern<<<(unsigned)grid, kS64Warps * 32, 0, s>>>(q, (const double*)hx, (const double*)hy, (const double*)u,
                                                   (const double*)p, (double*)v, (double*)u_next, o, scale);
  };
  if (many)
    store ? run(k_leapfrog64<FORM, true, true, true>) : run(k_leapfrog64<FORM, false, true, true>);
  else if (o.energy)
    store ? run(k_leapfrog64<FORM, true, true>) : run(k_leapfrog64<FORM, false, true>);
  else
    store ? run(k_leapfrog64<FORM, true, false>) : run(k_leapfrog64<FORM, false, false>);
  return cudaGetLastError();
}

}  // namespace

int step64_strips(int64_t nx) { return (int)((nx - 1 + kS64Out - 1) / kS64Out); }

// Rows per tile: the count (at most 32) that minimises the rows of the busiest of the 608
// schedulers, each tile charged one more for its first loads and flux.
int step64_rows(int64_t nx, int64_t ny) {
  const int64_t strips = step64_strips(nx), inner = ny - 2, slots = 152 * 4;
  int best = 1;
  int64_t least = INT64_MAX;
  for (int r = 1; r <= 32; ++r) {
    const int64_t tiles = strips * ((inner + r - 1) / r), busy = (tiles + slots - 1) / slots * (r + 1);
    if (busy <= least) {
      least = busy;
      best = r;
    }
  }
  return best;
}

int64_t step64_ctas(int64_t nx, int64_t ny, int rows) {
  if (rows <= 0) rows = step64_rows(nx, ny);
  return (step64_strips(nx) * ((ny - 2 + rows - 1) / rows) + kS64Warps - 1) / kS64Warps;
}

cudaError_t launch_step64(const StencilGeom& g, int form, const void* hx, const void* hy, const void* u_prev,
                          const void* u_cur, void* v, void* u_next, const PassOut& o, bool store, int rows,
                          cudaStream_t s) {
  return form == TSU_FORM_STANDARD ? step64<0>(g, hx, hy, u_prev, u_cur, v, u_next, o, store, rows, s)
                                   : step64<1>(g, hx, hy, v, u_cur, v, u_next, o, store, rows, s);
}

cudaError_t launch_energy64(const StencilGeom& g, const double* part, int64_t ncta, int64_t nsteps, double* energy,
                            cudaStream_t s) {
  k_energy64<<<(unsigned)nsteps, kS64Warps * 32, 0, s>>>(part, energy, g.dxdy / (2.0 * g.tau * g.tau), (int)ncta);
  return cudaGetLastError();
}

cudaError_t launch_adjoint64(const StencilGeom& g, const void* hx, const void* hy, const void* lam, void* lam_pp,
                             const void* u, void* gx, void* gy, const RecBuckets& rb, cudaStream_t s) {
  const S64Geom q = s64_geom(g, 0);
  k_adjoint64<<<(unsigned)((q.ntiles + kS64Warps - 1) / kS64Warps), kS64Warps * 32, 0, s>>>(
      q, (const double*)hx, (const double*)hy, (const double*)lam, (double*)lam_pp, (const double*)u, (double*)gx,
      (double*)gy, rb);
  return cudaGetLastError();
}

}  // namespace tsu
