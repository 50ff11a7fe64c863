// The step of small and medium lattices: one CTA per two-dimensional tile.
//
// The strip kernel marches each CTA up its rows, which streams a large
// lattice at the least traffic but takes a fixed chain of row iterations
// (load, barrier, mu, barrier, collide) one after another: with only a few
// CTAs that chain is the whole step.  Here a CTA takes a TW x TH tile at
// once: every population its nodes and their density frame pull is requested
// before the first is used, and the step is three phases with two barriers,
//   1. rho over the tile and two nodes around it      (shared memory)
//   2. mu over the tile and one node around it        (shared memory),
//      rho and grad rho of the own nodes              (registers)
//   3. grad mu, the collision and the stores,
// at the price of evaluating the frame's densities and chemical potentials
// again in every tile (0.41 times the tile's densities at 32 x 16, 0.56 at 16 x
// 16, 0.88 at 16 x 8, 2.0 at 8 x 4).  The chain of
// phases, not the traffic, bounds it up to about 256^2.  us per step with the
// strip kernel and here: FP64 4 x 256 48.9 and 5.1, 100^2 49.2 and 5.7, 256^2
// 51.2 and 17.4; FP32 100^2 8.1 and 2.0, 256^2 7.5 and 2.8, 512^2 8.7 and 5.4,
// 1023 x 771 19.9 and 12.0, 1024^2 18.3 and 14.3.  Each node goes through the same device functions in
// the same order as in the strip kernel, so the result is the same bit for
// bit.
#include <cuda_runtime.h>

#include <algorithm>

#include "lbm_kernels.cuh"
#include "strip_launch.cuh"

namespace wblbe {

namespace {

// Resident CTAs the register budget must allow (0: left to the compiler).  Left
// alone the FP64 pair of rows gets 80 registers; asked for four CTAs it gets 98
// to 102, and the fewer resident warps wait less for the FP64 pipe than the
// shorter live ranges cost; us per step before and after: well-balanced 256^2
// 18.2 and 17.4, 512^2 59.2 and 56.9, 1023 x 771 173.8 and 166.9, standard
// 18.9 and 17.5, 61.7 and 57.3, 181.5 and 168.0.  (1 gives the same code; 6, 80
// registers again, 17.8.)  The FP32 shapes are faster as they are: 1024^2 15.2,
// with 1 15.9.
template <typename T, int PR>
constexpr int min_ctas() {
  return sizeof(T) == 8 && PR == 2 ? 4 : 0;
}

// A thread owns PR nodes of one column (rows ty * PR ..); the TW * TH / PR
// owners come first, and the other threads of the CTA (if any) start on the
// frame, whose work would otherwise follow the owners' own.
template <typename T, int SCH, int MODE, int TW, int TH, int PR, int NT>
__global__ void __launch_bounds__(NT, min_ctas<T, PR>())
    lbm_tile_kernel(const T* src, T* dst, const KParams p, const MomentsOut mo) {
  static_assert(SCH == kSchStandard || SCH == kSchWB, "potential-form schemes");
  static_assert(sizeof(T) == 8 || PR == 2, "FP32 threads own a pair of rows");
  constexpr bool STATS = MODE != kModeStep;
  constexpr int FW = TW + 4, FH = TH + 4;       // the density frame
  constexpr int NO = TW * TH / PR;              // owner threads
  static_assert(NT >= NO && NT % 32 == 0 && TH % PR == 0 && TH % 2 == 0, "tile shape");
  __shared__ T rho_s[FH][FW], mu_s[FH][FW];     // [2 + row][2 + column] of the tile

  const int tid = threadIdx.x;
  const int x0 = blockIdx.x * TW, y0 = blockIdx.y * TH;
  const int nx = p.nx, ny = p.ny;
  const bool owner = tid < NO;
  const int tx = tid % TW, r0 = (tid / TW) * PR;
  const int first_halo = tid >= NO ? tid - NO : tid + NT - NO;

  auto ld = [&](int i, unsigned off) {
    return WB_IN(off, p.plane) ? (src + i * p.plane)[off] : T(0);
  };
  // f_i(x) = P_i(x - c_i) from the wrapped columns (west, own, east) and row
  // offsets (below, own, above)
  auto pull = [&](T(&g)[9], unsigned xw, unsigned xc, unsigned xe, unsigned rb, unsigned rc,
                  unsigned ra) {
    g[0] = ld(0, rc + xc);
    g[1] = ld(1, rc + xw);
    g[2] = ld(2, rb + xc);
    g[3] = ld(3, rc + xe);
    g[4] = ld(4, ra + xc);
    g[5] = ld(5, rb + xw);
    g[6] = ld(6, rb + xe);
    g[7] = ld(7, ra + xe);
    g[8] = ld(8, ra + xw);
  };
  auto rho_of = [](const T(&g)[9]) {
    if constexpr (sizeof(T) == 4)
      return g[0] + (((g[1] + g[3]) + (g[2] + g[4])) + ((g[5] + g[7]) + (g[6] + g[8])));
    else
      return ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8];
  };

  chain_wait();
  // ---- phase 1: densities ----
  T g[PR][9];
  if (owner) {
    const int xc = wrap_index(x0 + tx, nx);
    const int xw = xc == 0 ? nx - 1 : xc - 1, xe = xc == nx - 1 ? 0 : xc + 1;
    int yr = wrap_index(y0 + r0, ny);
    unsigned rb = (unsigned)((yr == 0 ? ny - 1 : yr - 1) * p.pitch);
    unsigned rc = (unsigned)(yr * p.pitch);
#pragma unroll
    for (int r = 0; r < PR; ++r) {
      yr = yr == ny - 1 ? 0 : yr + 1;
      const unsigned ra = (unsigned)(yr * p.pitch);
      pull(g[r], xw, xc, xe, rb, rc, ra);
      rb = rc;
      rc = ra;
    }
  }
  // the frame: two rows below, two above, then two columns on each side
  constexpr int kRowHalo = 2 * FW, kHaloN = 4 * FW + 4 * TH;
  for (int h = first_halo; h < kHaloN; h += NT) {
    int fx, fy;
    if (h < 2 * kRowHalo) {
      fy = h / FW;
      fx = h - fy * FW;
      if (fy >= 2) fy += TH;
    } else {
      const int q = h - 2 * kRowHalo;
      fy = 2 + (q >> 2);
      fx = q & 3;
      if (fx >= 2) fx += TW;
    }
    const int xc = wrap_index(x0 - 2 + fx, nx), yc = wrap_index(y0 - 2 + fy, ny);
    T f[9];
    pull(f, xc == 0 ? nx - 1 : xc - 1, xc, xc == nx - 1 ? 0 : xc + 1,
         (unsigned)((yc == 0 ? ny - 1 : yc - 1) * p.pitch), (unsigned)(yc * p.pitch),
         (unsigned)((yc == ny - 1 ? 0 : yc + 1) * p.pitch));
    if (WB_IN(fy, FH) && WB_IN(fx, FW)) rho_s[fy][fx] = rho_of(f);
  }
  T rs[PR];
  const int fx = 2 + tx, fy = 2 + r0;
  if (owner) {
#pragma unroll
    for (int r = 0; r < PR; ++r) {
      rs[r] = rho_of(g[r]);
      rho_s[fy + r][fx] = rs[r];
    }
  }
  __syncthreads();

  // ---- phase 2: chemical potential; grad rho of the own nodes ----
  const NodeConsts<T> cc = consts_of(p, T(0));
  const T two_beta = cc.two_beta, dl = cc.dl, dg = cc.dg, kappa6 = cc.kappa6;
  T mu[PR], grx[PR], gry[PR];
  if constexpr (sizeof(T) == 4) {
    const float2 tb2 = splat(two_beta), dl2 = splat(dl), dg2 = splat(dg), k62 = splat(kappa6);
    auto V = [](T lo, T hi) { return make_float2(lo, hi); };
    // mu at frame positions (ax, ay) and (bx, by), one per lane
    auto mu2 = [&](int ax, int ay, int bx, int by) {
      auto at = [&](int dx, int dy) { return V(rho_s[ay + dy][ax + dx], rho_s[by + dy][bx + dx]); };
      return chem_pot_x2(at(0, 0), at(1, 0), at(-1, 0), at(0, 1), at(0, -1), at(1, 1), at(-1, 1),
                         at(1, -1), at(-1, -1), tb2, dl2, dg2, k62);
    };
    if (owner) {
      const float2 m = mu2(fx, fy, fx, fy + 1);
      auto at = [&](int dx, int dy) { return V(rho_s[fy + dy][fx + dx], rho_s[fy + 1 + dy][fx + dx]); };
      float2 gx2, gy2;
      iso_grad_x2(at(1, 0), at(-1, 0), at(0, 1), at(0, -1), at(1, 1), at(-1, 1), at(1, -1),
                  at(-1, -1), gx2, gy2);
      mu_s[fy][fx] = mu[0] = m.x;
      mu_s[fy + 1][fx] = mu[1] = m.y;
      grx[0] = gx2.x;
      grx[1] = gx2.y;
      gry[0] = gy2.x;
      gry[1] = gy2.y;
    }
    // ring: the rows below and above (one per lane), then the two sides
    for (int h = first_halo; h < TW + 2 + TH; h += NT) {
      const int ax = h < TW + 2 ? 1 + h : 1, ay = h < TW + 2 ? 1 : h - TW;
      const int bx = h < TW + 2 ? 1 + h : TW + 2, by = h < TW + 2 ? TH + 2 : h - TW;
      const float2 m = mu2(ax, ay, bx, by);
      if (WB_IN(ay, FH) && WB_IN(ax, FW)) mu_s[ay][ax] = m.x;
      if (WB_IN(by, FH) && WB_IN(bx, FW)) mu_s[by][bx] = m.y;
    }
  } else {
    if (owner) {
      T c[PR + 2], ps[PR + 2], pd[PR + 2];
#pragma unroll
      for (int r = 0; r < PR + 2; ++r) {
        const T* row = rho_s[fy + r - 1];
        c[r] = row[fx];
        ps[r] = row[fx + 1] + row[fx - 1];
        pd[r] = row[fx + 1] - row[fx - 1];
      }
#pragma unroll
      for (int r = 0; r < PR; ++r) {
        mu[r] = chem_pot_rows(c[r + 1], ps[r + 1], c[r + 2], c[r], ps[r + 2], ps[r], two_beta,
                                 dl, dg, kappa6);
        iso_grad12_rows(pd[r + 1], pd[r + 2], pd[r], c[r + 2], c[r], ps[r + 2], ps[r], grx[r],
                           gry[r]);
        mu_s[fy + r][fx] = mu[r];
      }
    }
    for (int h = first_halo; h < 2 * (TW + 2) + 2 * TH; h += NT) {
      int hx, hy;
      if (h < 2 * (TW + 2)) {
        hx = 1 + (h >= TW + 2 ? h - (TW + 2) : h);
        hy = h >= TW + 2 ? TH + 2 : 1;
      } else {
        const int q = h - 2 * (TW + 2);
        hx = (q & 1) ? TW + 2 : 1;
        hy = 2 + (q >> 1);
      }
      const T *rn = rho_s[hy + 1], *rc = rho_s[hy], *rb = rho_s[hy - 1];
      if (WB_IN(hy, FH) && WB_IN(hx, FW))
        mu_s[hy][hx] = chem_pot(rc[hx], rc[hx + 1], rc[hx - 1], rn[hx], rb[hx], rn[hx + 1],
                                 rn[hx - 1], rb[hx + 1], rb[hx - 1], two_beta, dl, dg, kappa6);
    }
  }
  __syncthreads();

  // ---- phase 3: collision ----
  StatsAcc<T> acc;
  const int x = x0 + tx, y = y0 + r0;
  if (owner && x < nx && y < ny) {
    if constexpr (sizeof(T) == 4) {
      auto at = [&](int dx, int dy) {
        return make_float2(mu_s[fy + dy][fx + dx], mu_s[fy + 1 + dy][fx + dx]);
      };
      float2 gmx, gmy, ux, uy;
      iso_grad_x2(at(1, 0), at(-1, 0), at(0, 1), at(0, -1), at(1, 1), at(-1, 1), at(1, -1),
                  at(-1, -1), gmx, gmy);
      float2 g2[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) g2[i] = make_float2(g[0][i], g[1][i]);
      const uint32_t ht = step_key(p.step + (p.step_base ? *p.step_base : 0LL));
      const float2 rnd = pair_uniforms((uint32_t)y * (uint32_t)nx + (uint32_t)x, ht);
      collide_x2<SCH>(g2, make_float2(rs[0], rs[1]), gmx, gmy, make_float2(grx[0], grx[1]),
                      make_float2(gry[0], gry[1]), cc, ux, uy, rnd);
      const T gl[9] = {g2[0].x, g2[1].x, g2[2].x, g2[3].x, g2[4].x,
                       g2[5].x, g2[6].x, g2[7].x, g2[8].x};
      emit_node<T, MODE, false>(p, mo, dst, y, x, x, false, false, gl, rs[0], mu[0], ux.x, uy.x,
                                acc, STATS);
      if (y + 1 < ny) {
        const T gh[9] = {g2[0].y, g2[1].y, g2[2].y, g2[3].y, g2[4].y,
                         g2[5].y, g2[6].y, g2[7].y, g2[8].y};
        emit_node<T, MODE, false>(p, mo, dst, y + 1, x, x, false, false, gh, rs[1], mu[1], ux.y,
                                  uy.y, acc, STATS);
      }
    } else {
#pragma unroll
      for (int r = 0; r < PR; ++r) {
        if (y + r < ny) {
          const T *mn = mu_s[fy + r + 1], *mc = mu_s[fy + r], *mb = mu_s[fy + r - 1];
          T gmx, gmy, ux, uy;
          iso_grad12(mc[fx + 1], mc[fx - 1], mn[fx], mb[fx], mn[fx + 1], mn[fx - 1],
                        mb[fx + 1], mb[fx - 1], gmx, gmy);
          collide<T, SCH, 12>(g[r], rs[r], gmx, gmy, grx[r], gry[r], cc, ux, uy);
          emit_node<T, MODE, false>(p, mo, dst, y + r, x, x, false, false, g[r], rs[r], mu[r], ux,
                                    uy, acc, STATS);
        }
      }
    }
  }
  if (STATS && mo.partials)
    write_stats_record<NT>(acc, mo.partials +
                                    (size_t)(blockIdx.y * gridDim.x + blockIdx.x) * kStatRec);
  chain_signal();
}

// FP64 step of the smallest lattices, at most two 8 x 4 tiles per SM.  An FP64
// warp instruction occupies its SM sub-partition for 64 cycles however few of
// its lanes are active, so the time is the longest warp's instruction count,
// and the tile's arithmetic is dealt out to four warps: two hold the same 32
// nodes and take, one after another, {rho, momentum}, {mu, grad rho and 1/rho}
// and, after a common part, {rest and axis populations, diagonal ones}; the
// other two take the frame (rho) and its ring (mu).  About 70 instructions on
// the longest warp where one warp of lbm_tile_kernel has 111, but a fifth more
// in all: us per step there and here, 4 x 256 5.1 and 3.9, 96 x 100 (2 tiles on
// every SM) 5.3 and 4.9, 100^2 (3 on some) 5.6 and 6.2.
template <int SCH>
__global__ void __launch_bounds__(128)
    lbm_tile_split_kernel(const double* src, double* dst, const KParams p) {
  constexpr int TW = 8, TH = 4, FW = TW + 4, FH = TH + 4;
  static_assert(TW * TH == 32 && FW * FH - 32 == 64 && (TW + 2) * (TH + 2) - 32 <= 32,
                "a warp's nodes, two warps' frame and one warp's ring");
  __shared__ double rho_s[FH][FW], mu_s[FH][FW];
  __shared__ double part_s[5][32];              // jx, jy, 1/rho, 12 grad rho of each node
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int x0 = blockIdx.x * TW, y0 = blockIdx.y * TH;
  const int nx = p.nx, ny = p.ny;
  // frame position: the nodes (warps 0 and 1), or the two rows below and above
  // and the two columns on each side (warps 2 and 3)
  int fx, fy;
  if (wid < 2) {
    fx = 2 + lane % TW;
    fy = 2 + lane / TW;
  } else {
    const int h = (wid - 2) * 32 + lane;
    if (h < 4 * FW) {
      fy = h / FW;
      fx = h - fy * FW;
      if (fy >= 2) fy += TH;
    } else {
      const int q = h - 4 * FW;
      fy = 2 + (q >> 2);
      fx = q & 3;
      if (fx >= 2) fx += TW;
    }
  }
  const int xc = wrap_index(x0 - 2 + fx, nx), yc = wrap_index(y0 - 2 + fy, ny);
  const unsigned xw = xc == 0 ? nx - 1 : xc - 1, xe = xc == nx - 1 ? 0 : xc + 1;
  const unsigned rb = (unsigned)((yc == 0 ? ny - 1 : yc - 1) * p.pitch);
  const unsigned rc = (unsigned)(yc * p.pitch);
  const unsigned ra = (unsigned)((yc == ny - 1 ? 0 : yc + 1) * p.pitch);
  const NodeConsts<double>& cc = p.d;
  chain_wait();
  auto ld = [&](int i, unsigned off) {
    return WB_IN(off, p.plane) ? (src + i * p.plane)[off] : 0.0;
  };
  double g[9] = {ld(0, rc + xc), ld(1, rc + xw), ld(2, rb + xc), ld(3, rc + xe), ld(4, ra + xc),
                 ld(5, rb + xw), ld(6, rb + xe), ld(7, ra + xe), ld(8, ra + xw)};
  if (wid == 1) {
    double jx, jy;
    momentum_f64(g, jx, jy);
    part_s[0][lane] = jx;
    part_s[1][lane] = jy;
  } else {
    rho_s[fy][fx] = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8];
  }
  __syncthreads();
  if (wid == 1) {
    const double *rn = rho_s[fy + 1], *rm = rho_s[fy], *rs = rho_s[fy - 1];
    double gx, gy;
    iso_grad12_rows(rm[fx + 1] - rm[fx - 1], rn[fx + 1] - rn[fx - 1], rs[fx + 1] - rs[fx - 1],
                    rn[fx], rs[fx], rn[fx + 1] + rn[fx - 1], rs[fx + 1] + rs[fx - 1], gx, gy);
    part_s[2][lane] = recip(rm[fx]);
    part_s[3][lane] = gx;
    part_s[4][lane] = gy;
  } else if (wid == 0 || wid == 2) {
    int x = fx, y = fy;
    if (wid == 2) {                             // the ring: rows below and above, sides
      const int h = lane < 2 * (TW + 2) ? lane : min(lane - 2 * (TW + 2), 2 * TH - 1);
      if (lane < 2 * (TW + 2)) {
        x = 1 + (h >= TW + 2 ? h - (TW + 2) : h);
        y = h >= TW + 2 ? TH + 2 : 1;
      } else {
        x = (h & 1) ? TW + 2 : 1;
        y = 2 + (h >> 1);
      }
    }
    const double *rn = rho_s[y + 1], *rm = rho_s[y], *rs = rho_s[y - 1];
    mu_s[y][x] = chem_pot(rm[x], rm[x + 1], rm[x - 1], rn[x], rs[x], rn[x + 1], rn[x - 1],
                          rs[x + 1], rs[x - 1], cc.two_beta, cc.dl, cc.dg, cc.kappa6);
  }
  __syncthreads();
  const int x = x0 - 2 + fx, y = y0 - 2 + fy;
  if (wid < 2 && x < nx && y < ny) {
    const double *mn = mu_s[fy + 1], *mc = mu_s[fy], *mb = mu_s[fy - 1];
    double gmx, gmy, ux, uy;
    iso_grad12(mc[fx + 1], mc[fx - 1], mn[fx], mb[fx], mn[fx + 1], mn[fx - 1], mb[fx + 1],
               mb[fx - 1], gmx, gmy);
    const double rho = rho_s[fy][fx], jx = part_s[0][lane], jy = part_s[1][lane];
    const double inv = part_s[2][lane], grx = part_s[3][lane], gry = part_s[4][lane];
    const unsigned off = (unsigned)(y * p.pitch + x);
    const bool in = WB_IN(y, ny) && WB_IN(x, p.pitch);
    // each branch keeps only what its stores need
    if (wid == 0) {
      collide12_f64<SCH>(g, rho, jx, jy, inv, gmx, gmy, grx, gry, cc, ux, uy);
#pragma unroll
      for (int i = 0; i < 5; ++i)
        if (in) (dst + i * p.plane)[off] = g[i];
    } else {
      collide12_f64<SCH>(g, rho, jx, jy, inv, gmx, gmy, grx, gry, cc, ux, uy);
#pragma unroll
      for (int i = 5; i < 9; ++i)
        if (in) (dst + i * p.plane)[off] = g[i];
    }
  }
  chain_signal();
}

template <typename T, int SCH, int MODE, int TW, int TH, int PR, int NT>
cudaError_t launch_shape(const void* src, void* dst, const KParams& kp, const MomentsOut& mo,
                         cudaStream_t s, bool chained) {
  ChainedLaunch l(dim3((kp.nx + TW - 1) / TW, (kp.ny + TH - 1) / TH), NT, 0, s, chained);
  return cudaLaunchKernelEx(&l.cfg, lbm_tile_kernel<T, SCH, MODE, TW, TH, PR, NT>,
                            static_cast<const T*>(src), static_cast<T*>(dst), kp, mo);
}

// Tile shapes, smallest first (TW x TH, nodes per thread, threads), and the
// largest number of tiles each is chosen for; us per step, GB300:
//   FP64   8 x 4, 1,  96  up to 380 tiles: the FP64 chain of one node sets the
//                         time, so every node has its own lane and the frame
//                         other warps (4 x 256: 5.1, 16 x 8 5.9; 100^2: 5.7
//                         and 6.0; 128^2, 512 tiles: 6.5 and 6.0)
//         16 x 8, 1, 256  up to one tile per SM (128^2: 6.0, 16 x 16 10.7)
//         16 x 16, 2, 128 the rest: row sums shared by two rows (256^2: 17.4,
//                         16 x 8 18.6; 512^2: 56.9 and 60.8, 32 x 16 66.9)
//   FP32  16 x 8, 2, 192  up to three tiles per SM (128^2: 2.2, 32 x 16 2.7;
//                         256^2, 512 tiles: both 2.8)
//         32 x 16, 2, 256 the rest (512^2: 5.4, 16 x 8 6.3; 1024^2 14.3 and
//                         20.7, 64 x 16 15.7, 32 x 32 15.8)
// (The SM count is a constant here because it decides the number of records, and
// with it the workspace size that a caller asks for without a device.)
struct Shape { int tw, th; long long max_tiles; };
constexpr long long kSMs = 152, kAny = 1LL << 40;
constexpr Shape kShapes64[] = {{8, 4, 380}, {16, 8, kSMs}, {16, 16, kAny}};
constexpr Shape kShapes32[] = {{16, 8, 3 * kSMs}, {32, 16, kAny}};
// Above these many nodes the strip kernel reads less and is faster: FP64
// 1600 x 1500 486 us per step here and 531 there, 1900^2 734 and 743, 2048^2
// 844 and 833; FP32 1500^2 35.8 and 38.3, 2048^2 62.6 and 58.4.
constexpr long long kMaxNodes64 = 3610000, kMaxNodes32 = 3000000;
// The passes that reduce statistics change over earlier: one CTA sums the
// records, one per tile here and one per run of rows there.  us here and there,
// read back: FP64 step with statistics 1023 x 771 241 and 250, 1100^2 353 and
// 352, 1500^2 628 and 551; moments 1100^2 258 and 237, 1500^2 446 and 359; FP32
// moments 1000 x 900 60 and 54, step 53 and 52, 1500^2 100 and 74, 98 and 77.
constexpr long long kMaxStats64 = 1200000, kMaxStats32 = 800000;

long long tiles_of(const Shape& s, int nx, int ny) {
  return (long long)((nx + s.tw - 1) / s.tw) * ((ny + s.th - 1) / s.th);
}
int shape_of(bool fp64, int nx, int ny) {
  const Shape* s = fp64 ? kShapes64 : kShapes32;
  int k = 0;
  while (tiles_of(s[k], nx, ny) > s[k].max_tiles) ++k;
  return k;
}

template <int SCH, int MODE>
cudaError_t launch_mode_tile(bool fp64, const void* src, void* dst, const KParams& kp,
                             const MomentsOut& mo, cudaStream_t s, bool ch) {
  const int k = shape_of(fp64, kp.nx, kp.ny);
  if (fp64 && MODE == kModeStep && k == 0 && tiles_of(kShapes64[0], kp.nx, kp.ny) <= 2 * kSMs) {
    ChainedLaunch l(dim3((kp.nx + 7) / 8, (kp.ny + 3) / 4), 128, 0, s, ch);
    return cudaLaunchKernelEx(&l.cfg, lbm_tile_split_kernel<SCH>, static_cast<const double*>(src),
                              static_cast<double*>(dst), kp);
  }
  if (fp64) {
    switch (k) {
      case 0: return launch_shape<double, SCH, MODE, 8, 4, 1, 96>(src, dst, kp, mo, s, ch);
      case 1: return launch_shape<double, SCH, MODE, 16, 8, 1, 256>(src, dst, kp, mo, s, ch);
      default: return launch_shape<double, SCH, MODE, 16, 16, 2, 128>(src, dst, kp, mo, s, ch);
    }
  }
  if (k == 0) return launch_shape<float, SCH, MODE, 16, 8, 2, 192>(src, dst, kp, mo, s, ch);
  return launch_shape<float, SCH, MODE, 32, 16, 2, 256>(src, dst, kp, mo, s, ch);
}

template <int SCH>
cudaError_t launch_scheme_tile(bool fp64, int mode, const void* src, void* dst, const KParams& kp,
                               const MomentsOut& mo, cudaStream_t s, bool ch) {
  switch (mode) {
    case kModeStep: return launch_mode_tile<SCH, kModeStep>(fp64, src, dst, kp, mo, s, ch);
    case kModeMoments: return launch_mode_tile<SCH, kModeMoments>(fp64, src, dst, kp, mo, s, ch);
    case kModeStepStats:
      return launch_mode_tile<SCH, kModeStepStats>(fp64, src, dst, kp, mo, s, ch);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

bool tile_path(int sch, bool fp64, int mode, int nx, int ny) {
  const bool step = mode == kModeStep;
  const long long most = fp64 ? (step ? kMaxNodes64 : kMaxStats64)
                              : (step ? kMaxNodes32 : kMaxStats32);
  return (sch == kSchStandard || sch == kSchWB) && (long long)nx * ny <= most &&
         (ny + 3) / 4 <= 65535;
}

int tile_records(bool fp64, int nx, int ny) {
  if (!tile_path(kSchWB, fp64, kModeStepStats, nx, ny)) return 0;
  return (int)tiles_of((fp64 ? kShapes64 : kShapes32)[shape_of(fp64, nx, ny)], nx, ny);
}

cudaError_t launch_tile(int sch, bool fp64, int mode, const void* src, void* dst,
                        const KParams& kp, const MomentsOut& mo, cudaStream_t s, bool chained) {
  return sch == kSchWB ? launch_scheme_tile<kSchWB>(fp64, mode, src, dst, kp, mo, s, chained)
                       : launch_scheme_tile<kSchStandard>(fp64, mode, src, dst, kp, mo, s, chained);
}

// Lattices of few rows and many columns: their last row of tiles is mostly
// padding, which the strip kernel does not have.  us per step there and here:
// FP64 200000 x 2 348 and 121, 40000 x 4 75 and 58, 10000 x 2 25.3 and 17.2,
// 10000 x 4 25.5 and 26.7, 40000 x 8 95 and 102; FP32 200000 x 2 25 and 12.6,
// 40000 x 2 6.5 and 4.7, 25000 x 4 5.1 and 5.4, 80000 x 18 31.3 and 24.9, 80000 x
// 12 15.0 and 17.9.  Neither the row count nor the padding alone draws that
// line, so the two times are estimated (us; over 189 FP64 and 192 FP32 sizes of
// 1 to 49 rows and 1500 to 500000 columns the choice is never more than 3 %
// slower than the tiles, nor more than 17 % slower than the better kernel).
// stats: for the passes with statistics, which the strips do in a smaller part
// of their step's time, and whose final pass reads one record per CTA (moments
// FP64 20000 x 4 84 us on tiles, 72 on strips, FP32 40000 x 20 63 and 50).
// rows_per_cta: of the strip kernel's launch, 128 columns wide.
bool flat_takes_strips(bool fp64, bool stats, int nx, int ny, int rows_per_cta) {
  const int last = fp64 ? 2 : 1;
  if (ny >= 64 || shape_of(fp64, nx, ny) != last) return false;
  const Shape& t = (fp64 ? kShapes64 : kShapes32)[last];
  const int cols = (nx + t.tw - 1) / t.tw, whole = ny / t.th, rest = ny % t.th;
  const int strips = (nx + 127) / 128, runs = (ny + rows_per_cta - 1) / rows_per_cta;
  const int ctas = strips * runs, records = cols * (whole + (rest ? 1 : 0));
  auto waves = [](int n) { return (n + (int)kSMs - 1) / (int)kSMs; };
  if (fp64) {
    // bound by the FP64 pipes: a tile's time is its four-row groups', a strip
    // CTA's its rows', shared evenly by the SMs; a lone CTA waits for its chain
    const double tiles =
        3.0 + cols / (double)kSMs * (whole * 7.8 + (rest ? 3.0 + 1.2 * ((rest + 3) / 4) : 0.0));
    const int full = strips * (ny / rows_per_cta);          // CTAs with all their rows
    const double strip = std::max({5.0 + waves(ctas) * (3.0 + 4.0 * ny / runs),
                                   5.0 + waves(full) * (3.0 + 4.0 * rows_per_cta),
                                   7.6 + 4.8 * rows_per_cta});
    return stats ? 4.0 + 0.8 * strip < 0.97 * (tiles + 0.01 * (records - ctas))
                 : strip < 0.98 * tiles;
  }
  // bound by the requests in flight: a base per tile and a share per row; a base
  // per strip CTA and a share per pair of rows, after one CTA's own chain
  const double tiles = 1.5 + cols * (whole * 0.0066 + (rest ? 0.0036 + 0.00019 * rest : 0.0));
  const double strip = 2.0 + 0.7 * ((rows_per_cta + 1) / 2) +
                       ctas * (0.0028 + 0.00135 * (runs == 1 ? ny + (ny & 1) : ny / (double)runs));
  return stats ? 2.0 + 0.5 * strip < 0.97 * (tiles + 0.004 * (records - ctas))
               : strip < 0.98 * tiles;
}

unsigned int tile_bounds_errors(bool reset) { return read_bounds_errors(reset); }

}  // namespace wblbe
