// FP64 reverse steps on chip: the reverse sweep over one checkpoint segment in one cooperative launch
// (the recursion of k_adjoint.cu; tiling and exchange of k_step_res64.cu).
//
// One reverse step per launch (k_adjoint64) takes 6 to 8 us on small grids, of which the FP64 pipe works 2:
// launches come in multiples of 2.05 us, and every step reads and writes lam, both gradients and the
// faces.  Here a CTA keeps them all in registers for the segment; a step reads the stored state u^n (one
// step ahead) and the receivers' values, and exchanges the edge of lam.  Same operations in the same
// order as k_adjoint64, so the same bits.
#include <atomic>

#include "resident64.cuh"
#include "stencil_common.cuh"

namespace tsu {
namespace {
using namespace dev;

struct A64Args {
  int32_t nx, ny;
  int64_t ld;
  double cx, cy;
  const double* hx;
  const double* hy;
  double* lam;   // lam^{n+1} in, lam^{n+1-nsteps} out
  double* lpp;   // lam^{n+2} in, lam^{n+2-nsteps} out
  double* gx;
  double* gy;
  const double* u;  // u^n of the first step; u^{n-k} at u - k ustride
  int64_t ustride;
  int rows, nstrips, nchunks, nsteps;
  ulonglong2* col;
  ulonglong2* row;
  const int64_t* rec_idx;
  int32_t nrec;
  const double* g;  // g^n of the first step; g^{n-k} at g - k nrec
  PollLimit wait;
  uint32_t skew;  // added to the tags sent: 0 (test hook: a number that no reader waits for)
};

struct A64Smem {
  double xch[2][kR64Warps][2][32];  // first and last row of every warp, double buffered
  double g[2][kResMaxRec];          // the receivers' values of this step and the next
  int2 rec[kResMaxRec];             // (row << 8 | lane, receiver), in receiver order
  int nrec;
};

template <int R>
__global__ void __launch_bounds__(kR64Threads, 1) k_adjoint_res64(const A64Args a) {
  extern __shared__ __align__(16) unsigned char a64_raw[];
  A64Smem& sm = *reinterpret_cast<A64Smem*>(a64_raw);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int cta = blockIdx.x, ncta = gridDim.x, nsx = a.nstrips;
  const int chunk = cta / nsx, strip = cta - chunk * nsx;
  const int c = strip * kR64Out + lane;
  const int y0 = 1 + chunk * a.rows, y1 = min(y0 + a.rows, a.ny - 1), rows = y1 - y0;
  const int base = rows / kR64Warps, extra = rows - base * kR64Warps;
  const int cnt = base + (w < extra ? 1 : 0), r0 = w * base + min(w, extra), j0 = y0 + r0;
  const int wl = min(rows, kR64Warps) - 1;  // the last warp with rows
  const bool in = c < a.nx;
  const bool node = lane >= 1 && lane <= 30 && c <= a.nx - 2;
  const bool xface = node || (lane == 0 && strip == 0);  // owns the face right of its column
  const bool has_l = strip > 0, has_r = strip + 1 < nsx, has_d = chunk > 0, has_u = chunk + 1 < a.nchunks;
  auto at = [&](const double* f, int j) { return in ? __ldcg(f + (int64_t)j * a.ld + c) : 0.0; };

  double l[R], p[R], hx[R], hy[R], ax[R], ay[R], u[R + 1], hd = 0.0, below = 0.0, above = 0.0, ay0 = 0.0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    l[r] = p[r] = hx[r] = hy[r] = ax[r] = ay[r] = 0.0;
    if (r < cnt) {
      l[r] = at(a.lam, j0 + r);
      p[r] = node ? at(a.lpp, j0 + r) : 0.0;
      hx[r] = at(a.hx, j0 + r);
      hy[r] = at(a.hy, j0 + r);
      ax[r] = xface ? at(a.gx, j0 + r) : 0.0;
      ay[r] = node ? at(a.gy, j0 + r) : 0.0;
    }
  }
  const bool row1 = cnt > 0 && j0 == 1;  // also owns the faces between row 0 and row 1
  if (cnt > 0) {
    hd = at(a.hy, j0 - 1);
    below = at(a.lam, j0 - 1);
    above = at(a.lam, j0 + cnt);
    if (row1 && node) ay0 = at(a.gy, 0);
  }
  auto load_u = [&](const double* f) {  // rows j0 .. j0 + cnt (the boundary holds zeros)
#pragma unroll
    for (int r = 0; r <= R; ++r) u[r] = cnt > 0 && r <= cnt ? at(f, j0 + r) : 0.0;
  };
  load_u(a.u);
  // the tile's receivers, in receiver order (interior nodes only)
  if (w == 0) {
    int n = 0;
    for (int b = 0; b < a.nrec; b += 32) {
      int2 e = make_int2(0, b + lane);
      bool own = false;
      if (b + lane < a.nrec) {
        const int64_t v = a.rec_idx[b + lane];
        const int64_t j = v >= 0 && v < (int64_t)a.ny * a.ld ? v / a.ld : 0, i = v - j * a.ld;
        own = j >= y0 && j < y1 && i >= 1 && i <= a.nx - 2 && (i - 1) / kR64Out == strip;
        if (own) e.x = (int)(j << 8) | (int)(i - strip * kR64Out);
      }
      const unsigned m = __ballot_sync(0xffffffffu, own);
      if (own) sm.rec[n + __popc(m & ((1u << lane) - 1u))] = e;
      n += __popc(m);
    }
    if (lane == 0) sm.nrec = n;
  }
  __syncthreads();
  const int nrec = sm.nrec;
  bool mine = false;  // some receiver lies on this warp's rows
  for (int q = 0; q < nrec; ++q) {
    const int j = sm.rec[q].x >> 8;
    mine = mine || (j >= j0 && j < j0 + cnt);
  }
  auto load_g = [&](int k) {
    for (int q = tid; q < nrec; q += kR64Threads)
      sm.g[k & 1][q] = a.g[sm.rec[q].y - (int64_t)k * a.nrec];
  };
  load_g(0);
  __syncthreads();
  auto col_rim = [&](int q, int k, int side) { return a.col + (((int64_t)q * ncta + k) * 2 + side) * kR64Rows + r0; };
  auto row_rim = [&](int q, int k, int side) { return a.row + (((int64_t)q * ncta + k) * 2 + side) * 32 + lane; };
  bool dead = false;
  const double cx = a.cx, cy = a.cy, gwx = -a.cx, gwy = -a.cy;

  for (int n = 0; n < a.nsteps; ++n) {
    const bool last = n + 1 == a.nsteps;
    double gd = 0.0;
    if (cnt > 0) gd = __dmul_rn(hd, __dsub_rn(l[0], below));
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (r >= cnt) break;
      const double lc = l[r], ln = r + 1 < R ? (r + 1 < cnt ? l[r + 1 < R ? r + 1 : r] : above) : above;
      const double lr = __shfl_down_sync(0xffffffffu, lc, 1), ur = __shfl_down_sync(0xffffffffu, u[r], 1);
      const double dlx = __dsub_rn(lr, lc), dly = __dsub_rn(ln, lc);
      const double fr = __dmul_rn(hx[r], dlx), gu = __dmul_rn(hy[r], dly);
      const double fl = __shfl_up_sync(0xffffffffu, fr, 1);
      const double b = __fma_rn(cx, __dsub_rn(fr, fl), __dmul_rn(cy, __dsub_rn(gu, gd)));
      const double val = __dadd_rn(__fma_rn(2.0, lc, -p[r]), b);
      ax[r] = __fma_rn(gwx, __dmul_rn(dlx, __dsub_rn(ur, u[r])), ax[r]);
      ay[r] = __fma_rn(gwy, __dmul_rn(dly, __dsub_rn(u[r + 1], u[r])), ay[r]);
      if (r == 0 && row1) ay0 = __fma_rn(gwy, __dmul_rn(lc, u[0]), ay0);
      p[r] = lc;
      l[r] = node ? val : 0.0;
      gd = gu;
    }
    if (mine) {  // lam^n += g^n
      for (int q = 0; q < nrec; ++q) {
        const int e = sm.rec[q].x, k = (e >> 8) - j0;
        if (k < 0 || k >= cnt) continue;
        const double g = (e & 255) == lane ? sm.g[n & 1][q] : 0.0;
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (r == k && (e & 255) == lane) l[r] += g;
      }
    }
    if (last) break;
    load_u(a.u - (int64_t)(n + 1) * a.ustride);
    load_g(n + 1);
    const int q = n & 1;
    const uint32_t tag = (uint32_t)n + 1u;
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (r < cnt && ((lane == 1 && has_l) || (lane == 30 && has_r)))
        put64(col_rim(q, cta, lane == 30 ? 1 : 0) + r, l[r], tag + a.skew);
    double top = l[0];
#pragma unroll
    for (int r = 1; r < R; ++r)
      if (r < cnt) top = l[r];
    if (cnt > 0) {
      if (w == 0 && has_d) put64(row_rim(q, cta, 0), l[0], tag + a.skew);
      if (w == wl && has_u) put64(row_rim(q, cta, 1), top, tag + a.skew);
      sm.xch[q][w][0][lane] = l[0];
      sm.xch[q][w][1][lane] = top;
    }
    __syncthreads();
    if (cnt > 0) {
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
        if (edge && r < cnt) l[r] = get64(x[r], cs + r, tag, a.wait, dead);
      if (dn) below = get64(xd, ds, tag, a.wait, dead);
      if (up) above = get64(xu, us, tag, a.wait, dead);
      __syncwarp();
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (r < cnt) {
      const int64_t q = (int64_t)(j0 + r) * a.ld + c;
      if (node) {
        a.lam[q] = l[r];
        a.lpp[q] = p[r];
        a.gy[q] = ay[r];
      }
      if (xface) a.gx[q] = ax[r];
    }
  if (row1 && node) a.gy[c] = ay0;
}

using A64Kernel = void (*)(const A64Args);
struct A64Variant {
  int rows;  // per warp
  A64Kernel kern;
};
const A64Variant kA64Variants[] = {{1, k_adjoint_res64<1>}, {2, k_adjoint_res64<2>}, {3, k_adjoint_res64<3>},
                                   {4, k_adjoint_res64<4>}, {6, k_adjoint_res64<6>}, {8, k_adjoint_res64<8>}};
constexpr int kA64Num = (int)(sizeof kA64Variants / sizeof kA64Variants[0]);

// SMs that hold a CTA of every variant on this device (0: not available), once per device
std::atomic<int> g_a64_sms[64];
int a64_sms() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int v = g_a64_sms[dev].load();
  if (v != 0) return v > 0 ? v : 0;
  int nsm = 0, coop = 0;
  bool ok = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop != 0;
  for (int k = 0; ok && k < kA64Num; ++k) {
    int q = 0;
    ok = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&q, kA64Variants[k].kern, kR64Threads, sizeof(A64Smem)) ==
             cudaSuccess &&
         q >= 1;
  }
  (void)cudaGetLastError();  // a refused query leaves no error behind
  v = ok ? (nsm < kResMaxCtas ? nsm : kResMaxCtas) : -1;
  g_a64_sms[dev].store(v);
  return v > 0 ? v : 0;
}

}  // namespace

cudaError_t launch_adjoint_res64(const StencilGeom& g, const void* hx, const void* hy, void* lam, void* lam_pp,
                                 const void* u, int64_t ustride, void* gx, void* gy, int32_t nrec,
                                 const int64_t* rec_idx, const void* gv, int64_t nsteps, void* ws, cudaStream_t s,
                                 bool hold, bool* ran) {
  *ran = false;
  const int64_t sms = a64_sms(), strips = r64_strips(g.nx), inner = g.ny - 2;
  if (!ws || sms <= 0 || strips < 1 || strips > sms || g.ny >= 1 << 22 || nsteps < 2 || nsteps > 16384 ||
      nrec > kResMaxRec)
    return cudaSuccess;
  const int64_t rows = (inner + sms / strips - 1) / (sms / strips);
  int k = 0;
  while (k < kA64Num && kA64Variants[k].rows < (rows + kR64Warps - 1) / kR64Warps) ++k;
  if (k == kA64Num) return cudaSuccess;
  A64Args a{};
  a.nx = g.nx;
  a.ny = g.ny;
  a.ld = g.ld;
  a.cx = g.cx;
  a.cy = g.cy;
  a.hx = (const double*)hx;
  a.hy = (const double*)hy;
  a.lam = (double*)lam;
  a.lpp = (double*)lam_pp;
  a.gx = (double*)gx;
  a.gy = (double*)gy;
  a.u = (const double*)u;
  a.ustride = ustride;
  a.rows = (int)rows;
  a.nstrips = (int)strips;
  a.nchunks = (int)((inner + rows - 1) / rows);
  a.nsteps = (int)nsteps;
  a.col = (ulonglong2*)ws;
  a.row = a.col + (int64_t)2 * a.nstrips * a.nchunks * 2 * kR64Rows;
  a.rec_idx = rec_idx;
  a.nrec = nrec;
  a.g = (const double*)gv;
  a.wait = r64_limit(ws, hold);
  a.skew = hold ? 1u << 31 : 0u;
  // no value may carry a tag of an earlier launch
  cudaError_t e = cudaMemsetAsync(ws, 0, kR64RimBytes, s);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.nstrips * a.nchunks));
  cfg.blockDim = dim3(kR64Threads);
  cfg.dynamicSmemBytes = sizeof(A64Smem);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kA64Variants[k].kern, a);
  *ran = e == cudaSuccess;
  return e;
}

}  // namespace tsu
