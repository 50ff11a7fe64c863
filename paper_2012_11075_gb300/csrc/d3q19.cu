// The three-dimensional form of the well-balanced LBE (and of the standard
// LBE) on the D3Q19 lattice, in FP64 or FP32-shifted storage: the wblbe3_*
// part of include/wblbe.h.
//
// The paper builds the well-balanced scheme in D dimensions (Sec. III): the
// equilibrium of Eq. mFeq, F = -rho grad(mu) (Eq. mF) and the forcing term of
// Eq. mFi, whose isotropic term carries D; Sec. V notes the construction
// carries over to other lattice Boltzmann models.  Here D = 3 on D3Q19
// (c_0 = 0; six axis vectors, w = 1/18; twelve edge vectors, w = 1/36;
// w_0 = 1/3; cs^2 = 1/3), with the isotropic central stencils
// grad(phi) = 3 sum_i w_i c_i phi(x + c_i) and
// lap(phi) = 6 sum_i w_i (phi(x + c_i) - phi(x)).
//
// An FP32 step is two kernels (d3_density, d3_step_f32).  An FP64 step, and the
// moments of both, are three kernels on the caller's stream (the FP64 pipe is the limit,
// not memory traffic):
//   d3_density:   rho(x) = sum_i P_i(x - c_i)           (pull, Eq. rhoU)
//   d3_chem_pot:  mu = mu_0(rho) - kappa lap(rho)        (Sec. II)
//   d3_collide:   the pulled populations, grad rho and grad mu, the force,
//                 u, the equilibrium and forcing terms, and the BGK update
//                 (Eq. D2Q9), stored at x for the next pull.
// Layout: nineteen planes P_i[(z ny + y) pitch + x], pitch = nx rounded up
// to 16 elements, two buffers (ping-pong); the planes hold f_i - s_i, with
// s_i the well-balanced rho0 vector s_0 = -(1 - w_0) rho0, s_i = w_i rho0 (0
// for the standard scheme), plus in FP32 the scheme's rest equilibrium at
// rho_ref = rho_g; the update carries the shift unchanged.  The density and
// chemical-potential fields hold rho - rho_ref and mu in the storage type.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <new>

#include "../../include/wblbe.h"
#include "lbm_kernels.cuh"
#include "strip_launch.cuh"

using namespace wblbe;

namespace {

constexpr int kQ3 = 19;
constexpr int kBlock3 = 128;
constexpr size_t kAlign3 = 256;
constexpr long long kMaxPlane3 = (1LL << 32) - kBlock3;   // elements of a population plane

// D3Q19 in the order rest, 6 axis (+x, -x, +y, -y, +z, -z), 12 edges in
// opposite pairs ((1,1,0), (-1,-1,0)), ((1,-1,0), (-1,1,0)), ((1,0,1),
// (-1,0,-1)), ((1,0,-1), (-1,0,1)), ((0,1,1), (0,-1,-1)), ((0,1,-1), (0,-1,1)).
__host__ __device__ constexpr int cx3(int i) {
  return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13)
             ? 1 : ((i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0);
}
__host__ __device__ constexpr int cy3(int i) {
  return (i == 3 || i == 7 || i == 10 || i == 15 || i == 17)
             ? 1 : ((i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1 : 0);
}
__host__ __device__ constexpr int cz3(int i) {
  return (i == 5 || i == 11 || i == 14 || i == 15 || i == 18)
             ? 1 : ((i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1 : 0);
}
__host__ __device__ constexpr double w3(int i) {
  return i == 0 ? 1.0 / 3.0 : (i < 7 ? 1.0 / 18.0 : 1.0 / 36.0);
}

struct P3 {
  int nx, ny, nz, pitch;
  unsigned nodes;                  // nx ny nz
  long long plane;                 // elements per population plane / field
  double rho_ref;                  // storage shift density, 0 in FP64
  NodeConsts<double> d;            // the update's constants in both types
  NodeConsts<float> f;
  double kc72, kf288;              // -kforce/72, kforce/288 (update3_f64)
  long long step;                  // the step being taken (FP32 rounding draws)
};

// Mirror-symmetric sum of the eighteen moving populations: opposite pairs
// first, the axis pairs together and the edge pairs by plane, so that a
// reflection of any axis maps the grouping onto itself (mirror-image nodes
// round alike; the FP32 path).
template <typename T>
__device__ __forceinline__ T moving_sum3(const T (&g)[19]) {
  const T ax = ((g[1] + g[2]) + (g[3] + g[4])) + (g[5] + g[6]);
  const T xy = (g[7] + g[8]) + (g[9] + g[10]);
  const T xz = (g[11] + g[12]) + (g[13] + g[14]);
  const T yz = (g[15] + g[16]) + (g[17] + g[18]);
  return ax + ((xy + xz) + yz);
}

// A uniform draw in [0, 1) on a 2^-23 grid from the node key k and the step
// key ht (MurmurHash3's finalizer), for the rounding of the 2D kernel.
__device__ __forceinline__ float node_uniform(uint32_t k, uint32_t ht) {
  return __fsub_rn(__uint_as_float(0x3f800000u | (fmix32(k + ht) >> 9)), 1.0f);
}
__device__ __forceinline__ const NodeConsts<float>& consts3(const P3& p, float) { return p.f; }
__device__ __forceinline__ const NodeConsts<double>& consts3(const P3& p, double) { return p.d; }

struct Out3 {
  double* rho;                     // [nz][ny][nx] fields (may be null)
  double* ux;
  double* uy;
  double* uz;
  double* mu;
  double* partials;                // per-block stats records (may be null)
};

__device__ __forceinline__ int wrap3(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

__device__ __forceinline__ long long at3(const P3& p, int x, int y, int z) {
  return ((long long)z * p.ny + y) * p.pitch + x;
}

// Element offsets of a node's wrapped neighbour columns, rows and planes
// (below, own, above): 32 bits, a plane has at most kMaxPlane3 elements.
struct Nbr3 {
  unsigned x[3], y[3], z[3];
  __device__ __forceinline__ Nbr3(const P3& p, int xx, int yy, int zz) {
    const unsigned row = (unsigned)p.pitch, layer = row * (unsigned)p.ny;
    x[0] = (unsigned)(xx == 0 ? p.nx - 1 : xx - 1);
    x[1] = (unsigned)xx;
    x[2] = (unsigned)(xx == p.nx - 1 ? 0 : xx + 1);
    y[0] = row * (unsigned)(yy == 0 ? p.ny - 1 : yy - 1);
    y[1] = row * (unsigned)yy;
    y[2] = row * (unsigned)(yy == p.ny - 1 ? 0 : yy + 1);
    z[0] = layer * (unsigned)(zz == 0 ? p.nz - 1 : zz - 1);
    z[1] = layer * (unsigned)zz;
    z[2] = layer * (unsigned)(zz == p.nz - 1 ? 0 : zz + 1);
  }
  __device__ __forceinline__ unsigned at(int dx, int dy, int dz) const {
    return x[1 + dx] + y[1 + dy] + z[1 + dz];
  }
};

// Element `off` of a population plane or a field (checked in the bounds-checked
// build, as are the stores below).
template <typename T>
__device__ __forceinline__ T elem3_at(const T* plane, unsigned off, const P3& p) {
  return WB_IN(off, p.plane) ? plane[off] : T(0);
}

// The node of a thread of the density, chemical-potential and FP64 collision
// kernels.  Rows that are not whole blocks are numbered along x, then y, then z
// without a break at their ends: an FP64 warp instruction costs the same with
// any number of active lanes, and rows of 101 nodes in blocks of their own fill
// 79 % of them (FP64 101 x 67 x 75: 261 us per step, 209 this way; 130 x 60 x 40
// 165 and 133).  Whole blocks keep the grid's coordinates, without divisions.
template <bool FLAT>
__device__ __forceinline__ bool node_of(const P3& p, int& x, int& y, int& z) {
  const unsigned id = blockIdx.x * (unsigned)kBlock3 + threadIdx.x;
  if (!FLAT) {
    x = (int)id;
    y = blockIdx.y;
    z = blockIdx.z;
    return x < p.nx;
  }
  const unsigned row = id / (unsigned)p.nx, layer = row / (unsigned)p.ny;
  x = (int)(id - row * (unsigned)p.nx);
  y = (int)(row - layer * (unsigned)p.ny);
  z = (int)layer;
  return id < p.nodes;
}

// rho = sum_i f_i with f_i(x) = P_i(x - c_i): in FP64 summed from i = 0 to
// 18; in FP32 the stored deviation rs = rho - rho_ref = g_0 + the
// mirror-symmetric moving sum (the collision repeats that sum for the exact
// mass balance).
template <typename T, bool FLAT>
__global__ void __launch_bounds__(kBlock3) d3_density(const T* src, T* rho, const P3 p) {
  int x, y, z;
  const bool on = node_of<FLAT>(p, x, y, z);
  chain_wait();
  if (!on) return;
  const Nbr3 nb(p, x, y, z);
  T g[kQ3];
#pragma unroll
  for (int i = 0; i < kQ3; ++i)
    g[i] = elem3_at(src + i * p.plane, nb.at(-cx3(i), -cy3(i), -cz3(i)), p);
  T s;
  if (sizeof(T) == 8) {
    s = g[0];                                     // f_0 (c_0 = 0)
#pragma unroll
    for (int i = 1; i < kQ3; ++i) s += g[i];
  } else {
    s = g[0] + moving_sum3(g);
  }
  const unsigned k = nb.at(0, 0, 0);
  if (WB_IN(k, p.plane)) rho[k] = s;
  chain_signal();
}

// mu from the sums of the axis and edge neighbours' densities and the own
// one.  The FP32 functions of this file name each rounding (mu3,
// grad3_from, force3, update3_f32): a result then does not depend on which
// multiply-adds the compiler contracts in one kernel or another.
__device__ __forceinline__ double mu3(double ax, double ed, double c, const NodeConsts<double>& q) {
  const double lap = __fma_rn(1.0 / 3.0, __fma_rn(-6.0, c, ax),
                              __dmul_rn(1.0 / 6.0, __fma_rn(-12.0, c, ed)));
  const double a = __dadd_rn(c, q.dl), b = __dadd_rn(c, q.dg);
  return __fma_rn(__dmul_rn(__dmul_rn(q.two_beta, a), b), __dadd_rn(a, b),
                  -__dmul_rn(q.kappa, lap));
}
__device__ __forceinline__ float mu3(float ax, float ed, float c, const NodeConsts<float>& q) {
  const float lap = __fmaf_rn(1.0f / 3.0f, __fmaf_rn(-6.0f, c, ax),
                              __fmul_rn(1.0f / 6.0f, __fmaf_rn(-12.0f, c, ed)));
  const float a = __fadd_rn(c, q.dl), b = __fadd_rn(c, q.dg);
  return __fmaf_rn(__fmul_rn(__fmul_rn(q.two_beta, a), b), __fadd_rn(a, b),
                   -__fmul_rn(q.kappa, lap));
}

// mu = mu_0(rho) - kappa lap(rho), mu_0 = 2 beta a b (a + b), a = rho - rho_l,
// b = rho - rho_g (Eq. doubleWell), lap = 6 sum_i w_i (rho(x + c_i) - rho(x)).
// The field holds rho - rho_ref (rho_ref = 0 in FP64), which the Laplacian
// does not see and a, b take up through dl = rho_ref - rho_l, dg.
template <typename T, bool FLAT>
__global__ void __launch_bounds__(kBlock3) d3_chem_pot(const T* rho, T* mu, const P3 p) {
  int x, y, z;
  const bool on = node_of<FLAT>(p, x, y, z);
  chain_wait();
  if (!on) return;
  const Nbr3 nb(p, x, y, z);
  // sums of the axis and edge neighbours, then the centre's share taken off
  // once per sum (rather than from every neighbour): 6 (ax/18 + ed/36)
  auto nbr = [&](int i) { return elem3_at(rho, nb.at(cx3(i), cy3(i), cz3(i)), p); };
  T ax = nbr(1), ed = nbr(7);
#pragma unroll
  for (int i = 2; i < kQ3; ++i) {
    if (i == 7) continue;
    if (i < 7) ax += nbr(i); else ed += nbr(i);
  }
  const unsigned k = nb.at(0, 0, 0);
  if (WB_IN(k, p.plane)) mu[k] = mu3(ax, ed, rho[k], consts3(p, T(0)));
  chain_signal();
}

// 12 grad(phi) from v(dx, dy, dz) = phi(x + (dx, dy, dz)); see grad3x12.
template <typename T, typename V>
__device__ __forceinline__ void grad3_sums(const V& v, T& gx, T& gy, T& gz) {
  const T axx = v(1, 0, 0) - v(-1, 0, 0), axy = v(0, 1, 0) - v(0, -1, 0),
          axz = v(0, 0, 1) - v(0, 0, -1);
  const T exy1 = v(1, 1, 0) - v(-1, -1, 0), exy2 = v(1, -1, 0) - v(-1, 1, 0);
  const T exz1 = v(1, 0, 1) - v(-1, 0, -1), exz2 = v(1, 0, -1) - v(-1, 0, 1);
  const T eyz1 = v(0, 1, 1) - v(0, -1, -1), eyz2 = v(0, 1, -1) - v(0, -1, 1);
  gx = fma(T(2), axx, (exy1 + exy2) + (exz1 + exz2));
  gy = fma(T(2), axy, (exy1 - exy2) + (eyz1 + eyz2));
  gz = fma(T(2), axz, (exz1 - exz2) + (eyz1 - eyz2));
}
// 12 grad(phi) = 36 sum_i w_i c_i phi(x + c_i): 2 (axis differences) +
// (edge differences); the factor 1/12 is folded into the constants that
// use the gradients.
template <typename T>
__device__ __forceinline__ void grad3x12(const T* phi, const Nbr3& nb, const P3& p, T& gx, T& gy,
                                         T& gz) {
  grad3_sums<T>([&](int dx, int dy, int dz) { return elem3_at(phi, nb.at(dx, dy, dz), p); }, gx, gy,
                gz);
}

// One component of u = (j + F/2) / rho (Eq. rhoU) from 12 grad mu and 12 grad
// rho, inv = 1/rho: F = -rho grad mu (Eq. mF), plus cs^2 grad rho in the
// potential form of the standard scheme.
template <bool WB>
__device__ __forceinline__ double vel3(double j, double rho, double gm, double gr, double inv) {
  double s = __fma_rn(__dmul_rn(rho, -1.0 / 24.0), gm, j);
  if (!WB) s = __fma_rn(1.0 / 72.0, gr, s);
  return __dmul_rn(s, inv);
}
template <bool WB>
__device__ __forceinline__ float vel3(float j, float rho, float gm, float gr, float inv) {
  const float nr = __fmul_rn(rho, -1.0f / 12.0f);
  const float F = WB ? __fmul_rn(nr, gm) : __fmaf_rn(nr, gm, __fmul_rn(1.0f / 36.0f, gr));
  return __fmul_rn(__fmaf_rn(0.5f, F, j), inv);
}

// Momentum from the differences of opposite pairs (each edge difference
// serves two components).
template <typename T>
__device__ __forceinline__ void momentum3(const T (&g)[19], T& jx, T& jy, T& jz) {
  const T d12 = g[1] - g[2], d34 = g[3] - g[4], d56 = g[5] - g[6];
  const T d78 = g[7] - g[8], d910 = g[9] - g[10], d1112 = g[11] - g[12];
  const T d1314 = g[13] - g[14], d1516 = g[15] - g[16], d1718 = g[17] - g[18];
  jx = ((d12 + d78) + (d910 + d1112)) + d1314;
  jy = ((d34 + d78) - (d910 - d1516)) + d1718;
  jz = ((d56 + d1112) - (d1314 - d1516)) - d1718;
}

// ---- FP32 on pairs of nodes -------------------------------------------------
// (a pair's lanes are two nodes; every rounding is named, as in the scalar
// functions above, whose operations these are in the same order)
__device__ __forceinline__ float2 moving_sum3_x2(const float2 (&g)[19]) {
  const float2 ax = add2(add2(add2(g[1], g[2]), add2(g[3], g[4])), add2(g[5], g[6]));
  const float2 xy = add2(add2(g[7], g[8]), add2(g[9], g[10]));
  const float2 xz = add2(add2(g[11], g[12]), add2(g[13], g[14]));
  const float2 yz = add2(add2(g[15], g[16]), add2(g[17], g[18]));
  return add2(ax, add2(add2(xy, xz), yz));
}
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 mu3_x2(float2 ax, float2 ed, float2 c,
                                         const NodeConsts<float>& q) {
  const float2 lap = fma2(splat(1.0f / 3.0f), fma2(splat(-6.0f), c, ax),
                          mul2(splat(1.0f / 6.0f), fma2(splat(-12.0f), c, ed)));
  const float2 a = add2(c, splat(q.dl)), b = add2(c, splat(q.dg));
  return fma2(mul2(mul2(splat(q.two_beta), a), b), add2(a, b), neg2(mul2(splat(q.kappa), lap)));
}
// 12 grad(phi) of rows y and y + 1 from three shared-memory planes (below, at,
// above) at [y][x]
template <int W>
__device__ __forceinline__ void grad3_planes(const float (*b)[W], const float (*c)[W],
                                             const float (*a)[W], int x, int y, float2& gx,
                                             float2& gy, float2& gz) {
  auto v = [&](int dx, int dy, int dz) {
    const float(*r)[W] = dz < 0 ? b : (dz == 0 ? c : a);
    return make_float2(r[y + dy][x + dx], r[y + 1 + dy][x + dx]);
  };
  const float2 axx = sub2(v(1, 0, 0), v(-1, 0, 0)), axy = sub2(v(0, 1, 0), v(0, -1, 0)),
               axz = sub2(v(0, 0, 1), v(0, 0, -1));
  const float2 exy1 = sub2(v(1, 1, 0), v(-1, -1, 0)), exy2 = sub2(v(1, -1, 0), v(-1, 1, 0));
  const float2 exz1 = sub2(v(1, 0, 1), v(-1, 0, -1)), exz2 = sub2(v(1, 0, -1), v(-1, 0, 1));
  const float2 eyz1 = sub2(v(0, 1, 1), v(0, -1, -1)), eyz2 = sub2(v(0, 1, -1), v(0, -1, 1));
  gx = fma2(splat(2.0f), axx, add2(add2(exy1, exy2), add2(exz1, exz2)));
  gy = fma2(splat(2.0f), axy, add2(sub2(exy1, exy2), add2(eyz1, eyz2)));
  gz = fma2(splat(2.0f), axz, add2(sub2(exz1, exz2), sub2(eyz1, eyz2)));
}
// a x + b y + c z, the first product of the innermost sum fused
__device__ __forceinline__ float2 dot3_x2(float2 ax, float2 bx, float2 ay, float2 by, float2 az,
                                          float2 bz) {
  return fma2(az, bz, fma2(ax, bx, mul2(ay, by)));
}

// The FP32 update of a pair of nodes (the terms of update3_f64 below): rs the
// stored densities, (mx, my, mz) 12 grad mu, (rx, ry, rz) 12 grad rho; key_a,
// key_b the nodes' numbers and ht the step's key (the draws of the rest
// populations' roundings).
template <bool WB>
__device__ __forceinline__ void update3_x2(float2 (&g)[19], float2 rs, float2 mx, float2 my,
                                           float2 mz, float2 rx, float2 ry, float2 rz,
                                           const NodeConsts<float>& q, uint32_t key_a,
                                           uint32_t key_b, uint32_t ht) {
  const float2 om = splat(q.omega), keep = splat(q.keep), c36 = splat(1.0f / 36.0f);
  const float2 r = add2(rs, splat(q.rho_ref));
  const float2 nr = mul2(r, splat(-1.0f / 12.0f));
  auto force = [&](float2 gm, float2 gr) {
    return WB ? mul2(nr, gm) : fma2(nr, gm, mul2(c36, gr));
  };
  const float2 Fx = force(mx, rx), Fy = force(my, ry), Fz = force(mz, rz);
  const float2 d12 = sub2(g[1], g[2]), d34 = sub2(g[3], g[4]), d56 = sub2(g[5], g[6]);
  const float2 d78 = sub2(g[7], g[8]), d910 = sub2(g[9], g[10]), d1112 = sub2(g[11], g[12]);
  const float2 d1314 = sub2(g[13], g[14]), d1516 = sub2(g[15], g[16]), d1718 = sub2(g[17], g[18]);
  const float2 jx = add2(add2(add2(d12, d78), add2(d910, d1112)), d1314);
  const float2 jy = add2(sub2(add2(d34, d78), sub2(d910, d1516)), d1718);
  const float2 jz = sub2(sub2(add2(d56, d1112), sub2(d1314, d1516)), d1718);
  const float2 inv = make_float2(recip(r.x), recip(r.y)), half = splat(0.5f);
  const float2 ux = mul2(fma2(half, Fx, jx), inv), uy = mul2(fma2(half, Fy, jy), inv),
               uz = mul2(fma2(half, Fz, jz), inv);
  const float2 m_in = WB ? moving_sum3_x2(g) : make_float2(0.f, 0.f);
  const float2 Gx = WB ? fma2(c36, rx, Fx) : Fx;          // F + cs^2 grad rho
  const float2 Gy = WB ? fma2(c36, ry, Fy) : Fy;
  const float2 Gz = WB ? fma2(c36, rz, Fz) : Fz;
  const float2 orho = mul2(om, r);
  const float2 t = fma2(mul2(splat(-1.5f), orho), dot3_x2(ux, ux, uy, uy, uz, uz),
                        neg2(mul2(splat(__fmul_rn(3.0f, q.kf)), dot3_x2(ux, Gx, uy, Gy, uz, Gz))));
  float2 Ca, Ce;
  if (WB) {
    const float2 ku = mul2(splat(__fmul_rn(q.kf, 1.0f / 12.0f)), dot3_x2(ux, rx, uy, ry, uz, rz));
    Ca = mul2(splat(1.0f / 18.0f), t);
    Ce = mul2(c36, fma2(splat(1.5f), ku, t));
  } else {
    const float2 b = fma2(om, rs, t);
    Ca = mul2(splat(1.0f / 18.0f), b);
    Ce = mul2(c36, b);
  }
  const float2 Aa = mul2(splat(0.25f), orho), Ae = mul2(splat(0.125f), orho);
  const float2 kh = splat(__fmul_rn(0.5f, q.kf)), kq = splat(__fmul_rn(0.25f, q.kf));
  const float2 k6 = splat(__fmul_rn(q.kf, 1.0f / 6.0f));
  const float2 o6 = mul2(orho, splat(1.0f / 6.0f));
  const float2 Mx = fma2(k6, Fx, mul2(o6, ux));
  const float2 My = fma2(k6, Fy, mul2(o6, uy));
  const float2 Mz = fma2(k6, Fz, mul2(o6, uz));
  const float2 Key = mul2(kq, Gy), Kez = mul2(kq, Gz);
  auto axis = [&](int i, int j, float2 cu, float2 G, float2 M) {
    const float2 E = fma2(cu, fma2(kh, G, mul2(Aa, cu)), Ca);
    g[i] = fma2(keep, g[i], add2(E, M));
    g[j] = fma2(keep, g[j], sub2(E, M));
    return E;
  };
  auto edge = [&](int i, int j, float2 cu, float2 K, float2 S) {
    const float2 E = fma2(cu, fma2(Ae, cu, K), Ce);
    g[i] = fma2(keep, g[i], fma2(half, S, E));
    g[j] = fma2(keep, g[j], fma2(splat(-0.5f), S, E));
    return E;
  };
  const float2 Ea1 = axis(1, 2, ux, Gx, Mx);
  const float2 Ea2 = axis(3, 4, uy, Gy, My);
  const float2 Ea3 = axis(5, 6, uz, Gz, Mz);
  const float2 Ee1 = edge(7, 8, add2(ux, uy), fma2(kq, Gx, Key), add2(Mx, My));
  const float2 Ee2 = edge(9, 10, sub2(ux, uy), fma2(kq, Gx, neg2(Key)), sub2(Mx, My));
  const float2 Ee3 = edge(11, 12, add2(ux, uz), fma2(kq, Gx, Kez), add2(Mx, Mz));
  const float2 Ee4 = edge(13, 14, sub2(ux, uz), fma2(kq, Gx, neg2(Kez)), sub2(Mx, Mz));
  const float2 Ee5 = edge(15, 16, add2(uy, uz), add2(Key, Kez), add2(My, Mz));
  const float2 Ee6 = edge(17, 18, sub2(uy, uz), sub2(Key, Kez), sub2(My, Mz));
  if (WB) {
    // The collision conserves the node's mass, so the rest population
    // follows from the balance: g_0' = g_0 + omega m_in - 2 sum E (the
    // moving ones leave as keep g + E +- O).  Its small one-signed O(u^2)
    // part would be lost in rounding g_0 ~ rho - rho_ref to float; TwoSum
    // keeps the remainder and a zero-mean rounding, seeded by the node and
    // the step, takes it into account.
    const float2 sE = add2(add2(add2(Ea1, Ea2), Ea3),
                           add2(add2(add2(Ee1, Ee2), add2(Ee3, Ee4)), add2(Ee5, Ee6)));
    float2 hsum, err;
    two_sum2(g[0], fma2(splat(-2.0f), sE, mul2(om, m_in)), hsum, err);
    g[0] = round_stochastic2(hsum, err,
                             make_float2(node_uniform(key_a, ht), node_uniform(key_b, ht)));
  } else {
    g[0] = sub2(rs, moving_sum3_x2(g));        // the standard scheme: the mass balance
  }
}

// The FP64 update of one node's populations.  For an opposite pair (i, i') the
// even part E and the odd part O of omega f^eq + kforce F_i are shared,
// g_i' = keep g_i + E + O, g_i'' = keep g_i' + E - O, with
//   E = w (9 (c.u)(c.A) - 3 S + kforce h (u.grad rho)) [+ omega w rho, standard],
//   O = 3 w c.M,   A = (omega rho / 2) u + kforce G,   S = u.A,
//   M = omega rho u + kforce F,
// G = F + cs^2 grad rho and h = (3|c|^2 - 3)/2 (Eq. mFi, D = 3) for the
// well-balanced scheme, G = F and h = 0 for the standard one (Eq. Fi).  On an
// axis (c.u)(c.A) is a product P = u_a A_a, on an edge (a, b) it is
// P_a + P_b +- X_ab with X_ab = u_a A_b + u_b A_a, and P_a + P_b = S - P_c, so
// u.u and u.G are not needed.  A, P, S, X, kforce F and omega rho are carried
// divided by 6: E_axis = 3 P - S, E_edge = S - 3/2 P_c + B +- 3/2 X,
// B = kforce (u.grad rho) / 24, O_axis = M, O_edge = (M_a +- M_b) / 2.
// 161 FP64 operations with both gradients (191 with u.u, u.G and the pairs'
// sums formed one by one); the FP64 pipe is what bounds the kernel.  128^3
// well-balanced: 940 us per step before, 824 us; errors against 128-bit
// arithmetic as before (WB: populations 0.8e-16 to 1.9e-16 relative).
template <bool WB>
__device__ __forceinline__ void update3_f64(double (&g)[19], double r, double gmx, double gmy,
                                            double gmz, double grx, double gry, double grz,
                                            double ux, double uy, double uz,
                                            const P3& p) {
  const NodeConsts<double>& q = p.d;
  const double kc = __dmul_rn(r, p.kc72), keep = q.keep;
  auto kforce = [&](double gm, double gr) {             // kforce F / 6
    return WB ? __dmul_rn(kc, gm) : __fma_rn(kc, gm, __dmul_rn(q.kf216, gr));
  };
  const double kFx = kforce(gmx, grx), kFy = kforce(gmy, gry), kFz = kforce(gmz, grz);
  const double kGx = WB ? __fma_rn(q.kf216, grx, kFx) : kFx;
  const double kGy = WB ? __fma_rn(q.kf216, gry, kFy) : kFy;
  const double kGz = WB ? __fma_rn(q.kf216, grz, kFz) : kFz;
  const double orho = __dmul_rn(q.omega, r);
  const double o6 = __dmul_rn(orho, 1.0 / 6.0), h6 = __dmul_rn(orho, 1.0 / 12.0);
  const double Ax = __fma_rn(h6, ux, kGx), Ay = __fma_rn(h6, uy, kGy), Az = __fma_rn(h6, uz, kGz);
  const double Mx = __fma_rn(o6, ux, kFx), My = __fma_rn(o6, uy, kFy), Mz = __fma_rn(o6, uz, kFz);
  const double Px = __dmul_rn(ux, Ax), Py = __dmul_rn(uy, Ay), Pz = __dmul_rn(uz, Az);
  const double S = __dadd_rn(__dadd_rn(Px, Py), Pz);
  double Ca, Ce;
  if (WB) {
    const double D = __fma_rn(uz, grz, __fma_rn(ux, grx, __dmul_rn(uy, gry)));
    Ca = -S;
    Ce = __fma_rn(p.kf288, D, S);
    // E_0 = omega rho - 6 (S + 2 B): rest equilibrium rho - (rho/2) u.u, F_0 of Eq. mFi
    g[0] = __fma_rn(keep, g[0], __fma_rn(-6.0, __fma_rn(2.0, Ce, -S), orho));
  } else {
    Ca = __fma_rn(1.0 / 18.0, orho, -S);
    Ce = __fma_rn(1.0 / 36.0, orho, S);
    g[0] = __fma_rn(keep, g[0], __dmul_rn(6.0, Ca));
  }
  auto axis = [&](int i, int j, double P, double M) {
    const double E = __fma_rn(3.0, P, Ca);
    g[i] = __fma_rn(keep, g[i], __dadd_rn(E, M));
    g[j] = __fma_rn(keep, g[j], __dadd_rn(E, -M));
  };
  // the four pairs of the edges in the plane of components a, b (P: the
  // third component's product)
  auto edges = [&](int i, int j, int k, int l, double ua, double Aa, double ub, double Ab, double P,
                   double Ma, double Mb) {
    const double X = __fma_rn(ua, Ab, __dmul_rn(ub, Aa)), E0 = __fma_rn(-1.5, P, Ce);
    const double Ep = __fma_rn(1.5, X, E0), Em = __fma_rn(-1.5, X, E0);
    const double Tp = __dadd_rn(Ma, Mb), Tm = __dadd_rn(Ma, -Mb);
    g[i] = __fma_rn(keep, g[i], __fma_rn(0.5, Tp, Ep));
    g[j] = __fma_rn(keep, g[j], __fma_rn(-0.5, Tp, Ep));
    g[k] = __fma_rn(keep, g[k], __fma_rn(0.5, Tm, Em));
    g[l] = __fma_rn(keep, g[l], __fma_rn(-0.5, Tm, Em));
  };
  axis(1, 2, Px, Mx);
  axis(3, 4, Py, My);
  axis(5, 6, Pz, Mz);
  edges(7, 8, 9, 10, ux, Ax, uy, Ay, Pz, Mx, My);
  edges(11, 12, 13, 14, ux, Ax, uz, Az, Py, Mx, Mz);
  edges(15, 16, 17, 18, uy, Ay, uz, Az, Px, My, Mz);
}

// One node: its pulled populations, 12 grad mu, 12 grad rho and u.
template <typename T, bool WB>
struct Node3 {
  T g[kQ3], rs, r, gmx, gmy, gmz, grx, gry, grz, ux, uy, uz;
  __device__ __forceinline__ Node3(const T* src, const T* rho, const T* mu, const P3& p,
                                   const Nbr3& nb) {
#pragma unroll
    for (int i = 0; i < kQ3; ++i)
      g[i] = elem3_at(src + i * p.plane, nb.at(-cx3(i), -cy3(i), -cz3(i)), p);
    rs = elem3_at(rho, nb.at(0, 0, 0), p);     // rho - rho_ref (rho in FP64)
    r = sizeof(T) == 4 ? rs + consts3(p, T(0)).rho_ref : rs;
    grad3x12<T>(mu, nb, p, gmx, gmy, gmz);
    grad3x12<T>(rho, nb, p, grx, gry, grz);
    T jx, jy, jz;
    momentum3(g, jx, jy, jz);
    const T inv = recip(r);
    ux = vel3<WB>(jx, r, gmx, grx, inv);
    uy = vel3<WB>(jy, r, gmy, gry, inv);
    uz = vel3<WB>(jz, r, gmz, grz, inv);
  }
};

// FP64 step: the collision of one node, and its stores.
template <bool WB, bool FLAT>
__global__ void __launch_bounds__(kBlock3) d3_collide(const double* src, double* dst,
                                                      const double* rho, const double* mu,
                                                      const P3 p) {
  int x, y, z;
  const bool on = node_of<FLAT>(p, x, y, z);
  chain_wait();
  if (!on) return;
  const Nbr3 nb(p, x, y, z);
  Node3<double, WB> n(src, rho, mu, p, nb);
  update3_f64<WB>(n.g, n.r, n.gmx, n.gmy, n.gmz, n.grx, n.gry, n.grz, n.ux, n.uy, n.uz, p);
  const unsigned k = nb.at(0, 0, 0);
#pragma unroll
  for (int i = 0; i < kQ3; ++i)
    if (WB_IN(k, p.plane)) (dst + i * p.plane)[k] = n.g[i];
  chain_signal();
}

// Fields and statistics of `planes` planes per CTA: one record for all of them,
// so that the reduction's shuffles and the final pass over the records (one
// CTA) are shared by several nodes of each thread.
template <typename T, bool WB>
__global__ void __launch_bounds__(kBlock3) d3_moments(const T* src, const T* rho, const T* mu,
                                                      const P3 p, const Out3 out, int planes) {
  const int x = blockIdx.x * kBlock3 + threadIdx.x, y = blockIdx.y;
  const int z0 = blockIdx.z * planes, z1 = min(z0 + planes, p.nz);
  StatsAcc<T> acc;
  chain_wait();
  for (int z = z0; z < z1 && x < p.nx; ++z) {
    const Nbr3 nb(p, x, y, z);
    const Node3<T, WB> n(src, rho, mu, p, nb);
    const double rd = sizeof(T) == 4 ? widen(n.rs) + p.rho_ref : (double)n.r;
    const double ux = widen(n.ux), uy = widen(n.uy), uz = widen(n.uz);
    const T muc = elem3_at(mu, nb.at(0, 0, 0), p);
    const size_t k = ((size_t)z * p.ny + y) * p.nx + x;
    if (WB_IN(k, p.nodes)) {
      if (out.rho) out.rho[k] = rd;
      if (out.ux) out.ux[k] = ux;
      if (out.uy) out.uy[k] = uy;
      if (out.uz) out.uz[k] = uz;
      if (out.mu) out.mu[k] = widen(muc);
    }
    acc.add(rd, muc, __fma_rn(uz, uz, __fma_rn(ux, ux, __dmul_rn(uy, uy))));
  }
  write_stats_record<kBlock3>(
      acc, out.partials + (size_t)((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) *
                              kStatRec);
}

// The FP32 step after the density: a CTA owns TX x TY columns and marches a
// run of planes along z; a thread owns two rows of a column, whose arithmetic
// runs on packed pairs.  Per plane, with the front plane f:
//   A. rho of plane f over the tile and two columns around it, read from the
//      density field into a ring of planes (the next plane's values are
//      requested an iteration ahead);
//   B. mu of plane f - 1 over the tile and one column around it, into a second
//      ring; rho and grad rho of the own nodes stay in registers; the
//      populations of plane f - 2 are requested before the arithmetic;
//   C. grad mu, the collision and the stores of plane f - 2.
// With the density kernel a step moves 236 bytes per update at DRAM speed
// (256^3: 94 % of the measured copy bandwidth; 152 algorithmic).  us per step
// of the three kernels before and of the two, well-balanced: 256^3 985 and 633,
// 192^3 463 and 283, 128^3 130 and 90, 101 x 67 x 75 42 and 29, 64^3 27 and
// 16.5.  Measured and not kept, 256^3: the density formed here too, from the
// populations of the tile and its frame (152 bytes from DRAM, the rest from
// L2; bound by the latency of its pulls), 716; the same with one node per
// thread 782, with all pulls of an iteration at once 844, with populations
// staged by 4-byte asynchronous copies 1178; three resident CTAs 663, five 689.
constexpr int kTX3 = 32, kTY3 = 8, kNT3 = kTX3 * kTY3 / 2;
constexpr int kMinB3 = 4;          // resident CTAs (128 registers)

template <bool WB>
__global__ void __launch_bounds__(kNT3, kMinB3)
    d3_step_f32(const float* src, float* dst, const float* rho, const P3 p, int run) {
  constexpr int TX = kTX3, TY = kTY3;
  constexpr int FW = TX + 4, FH = TY + 4, MW = TX + 2, MH = TY + 2;
  __shared__ float rho_s[4][FH][FW];           // [f & 3][2 + y][2 + x]
  __shared__ float mu_s[4][MH][MW];            // [f & 3][1 + y][1 + x]
  const int tid = threadIdx.x, tx = tid % TX, ty = 2 * (tid / TX);
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  const int z0 = blockIdx.z * run, z1 = min(z0 + run, p.nz);
  chain_wait();

  // element offsets of a column's west, own and east elements and of four
  // rows: below the pair, the pair, above it
  struct Col { unsigned x[3], y[4]; };
  auto column = [&](int x, int y) {
    Col c;
    const int xc = wrap_index(x, p.nx);
    c.x[0] = (unsigned)(xc == 0 ? p.nx - 1 : xc - 1);
    c.x[1] = (unsigned)xc;
    c.x[2] = (unsigned)(xc == p.nx - 1 ? 0 : xc + 1);
    int yr = wrap_index(y - 1, p.ny);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      c.y[k] = (unsigned)p.pitch * (unsigned)yr;
      yr = yr == p.ny - 1 ? 0 : yr + 1;
    }
    return c;
  };
  const Col own = column(x0 + tx, y0 + ty);
  // the frame in pairs of rows: the two rows below, the two above, and two
  // columns on each side
  constexpr int kFrame = 2 * FW + 2 * TY;
  const bool has_frame = tid < kFrame;
  static_assert(kFrame <= kNT3, "one pair of the frame per thread");
  int hx, hy;
  if (tid < 2 * FW) {
    hx = tid < FW ? tid : tid - FW;
    hy = tid < FW ? 0 : TY + 2;
  } else {
    const int k = tid - 2 * FW;
    hx = (k & 3) < 2 ? (k & 3) : TX + (k & 3);
    hy = 2 + 2 * (k >> 2);
  }
  const Col frame = column(x0 - 2 + hx, y0 - 2 + hy);
  // mu's ring: the rows below and above (one per lane), then the two sides
  constexpr int kRing = MW + TY;
  static_assert(kRing <= kNT3, "one pair of the ring per thread");
  const bool has_ring = tid < kRing;
  const bool rows = tid < MW;
  const int rax = rows ? tid : 0, ray = rows ? 0 : 1 + tid - MW;
  const int rbx = rows ? tid : MW - 1, rby = rows ? MH - 1 : 1 + tid - MW;

  // g_i(x) = P_i(x - c_i) of a pair of rows; z: offsets of the planes below,
  // at and above
  auto pull = [&](float2(&g)[19], const Col& c, unsigned zb, unsigned zc, unsigned za) {
#pragma unroll
    for (int i = 0; i < kQ3; ++i) {
      const unsigned xz = (cz3(i) == 1 ? zb : (cz3(i) == 0 ? zc : za)) + c.x[1 - cx3(i)];
      const float* pl = src + i * p.plane;
      g[i] = make_float2(elem3_at(pl, xz + c.y[1 - cy3(i)], p), elem3_at(pl, xz + c.y[2 - cy3(i)], p));
    }
  };
  const unsigned layer = (unsigned)p.pitch * (unsigned)p.ny;
  auto zoff = [&](int z) { return layer * (unsigned)wrap_index(z, p.nz); };
  int f = z0 - 2;
  // planes f - 3 .. f + 1
  unsigned zm3 = 0, zm2 = 0, zm1 = zoff(f - 1), zc = zoff(f), zp = zoff(f + 1);
  int znext = wrap_index(f + 1, p.nz);

  const NodeConsts<float> q = p.f;
  const uint32_t ht = step_key(p.step);
  const bool mine_a = x0 + tx < p.nx && y0 + ty < p.ny, mine_b = mine_a && y0 + ty + 1 < p.ny;
  const float2 zero = make_float2(0.f, 0.f);
  float2 prs = zero, pgx = zero, pgy = zero, pgz = zero;   // rho - rho_ref, 12 grad rho of f - 2
  auto ld2 = [&](const Col& c, unsigned z) {
    return make_float2(elem3_at(rho, z + c.y[1] + c.x[1], p), elem3_at(rho, z + c.y[2] + c.x[1], p));
  };
  float2 nr = ld2(own, zc), nh = has_frame ? ld2(frame, zc) : zero;
  for (; f < z1 + 2; ++f) {
    const int c = f - 2;                        // the plane to collide
    const bool upd = mine_a && c >= z0;
    rho_s[f & 3][2 + ty][2 + tx] = nr.x;
    rho_s[f & 3][3 + ty][2 + tx] = nr.y;
    if (has_frame && WB_IN(hy, FH - 1) && WB_IN(hx, FW)) {
      rho_s[f & 3][hy][hx] = nh.x;
      rho_s[f & 3][hy + 1][hx] = nh.y;
    }
    if (f + 1 < z1 + 2) {
      nr = ld2(own, zp);
      if (has_frame) nh = ld2(frame, zp);
    }
    __syncthreads();
    float2 g[19];
    if (upd) pull(g, own, zm3, zm2, zm1);
    float2 rs = zero, gx = zero, gy = zero, gz = zero;
    if (f >= z0) {
      const float(*rb)[FW] = rho_s[(f + 2) & 3], (*rc)[FW] = rho_s[(f + 3) & 3],
                 (*ra)[FW] = rho_s[f & 3];
      // mu at two nodes of the frame, from the neighbours' sums in the
      // direction order of d3_chem_pot
      auto mu_at = [&](int ax, int ay, int bx, int by) {
        auto v = [&](int dx, int dy, int dz) {
          const float(*r)[FW] = dz < 0 ? rb : (dz == 0 ? rc : ra);
          return make_float2(r[ay + dy][ax + dx], r[by + dy][bx + dx]);
        };
        float2 sa = v(1, 0, 0), se = v(1, 1, 0);
#pragma unroll
        for (int i = 2; i < 7; ++i) sa = add2(sa, v(cx3(i), cy3(i), cz3(i)));
#pragma unroll
        for (int i = 8; i < kQ3; ++i) se = add2(se, v(cx3(i), cy3(i), cz3(i)));
        return mu3_x2(sa, se, v(0, 0, 0), q);
      };
      const int x = 2 + tx, y = 2 + ty;
      const float2 m = mu_at(x, y, x, y + 1);
      mu_s[(f + 3) & 3][1 + ty][1 + tx] = m.x;
      mu_s[(f + 3) & 3][2 + ty][1 + tx] = m.y;
      rs = make_float2(rc[y][x], rc[y + 1][x]);
      grad3_planes(rb, rc, ra, x, y, gx, gy, gz);
      if (has_ring) {
        const float2 h = mu_at(rax + 1, ray + 1, rbx + 1, rby + 1);
        if (WB_IN(ray, MH) && WB_IN(rax, MW)) mu_s[(f + 3) & 3][ray][rax] = h.x;
        if (WB_IN(rby, MH) && WB_IN(rbx, MW)) mu_s[(f + 3) & 3][rby][rbx] = h.y;
      }
    }
    __syncthreads();
    if (upd) {
      float2 mx, my, mz;
      grad3_planes(mu_s[(f + 1) & 3], mu_s[(f + 2) & 3], mu_s[(f + 3) & 3], 1 + tx, 1 + ty, mx, my,
                   mz);
      const uint32_t key = (uint32_t)(((long long)c * p.ny + y0 + ty) * p.nx + x0 + tx);
      update3_x2<WB>(g, prs, mx, my, mz, pgx, pgy, pgz, q, key, key + (uint32_t)p.nx, ht);
      const unsigned ka = zm2 + own.x[1] + own.y[1], kb = zm2 + own.x[1] + own.y[2];
      float *da = dst + ka, *db = dst + kb;
      const bool in_a = WB_IN(ka, p.plane), in_b = mine_b && WB_IN(kb, p.plane);
#pragma unroll
      for (int i = 0; i < kQ3; ++i) {
        if (in_a) da[i * p.plane] = g[i].x;
        if (in_b) db[i * p.plane] = g[i].y;
      }
    }
    prs = rs;
    pgx = gx;
    pgy = gy;
    pgz = gz;
    zm3 = zm2;
    zm2 = zm1;
    zm1 = zc;
    zc = zp;
    znext = znext == p.nz - 1 ? 0 : znext + 1;
    zp = layer * (unsigned)znext;
  }
  chain_signal();
}

// f = f^eq(rho, 0) stored for the pull: P_i(x) = f_i^eq(rho(x + c_i)) - s_i.
template <typename T>
__global__ void d3_init(const double* __restrict__ rho_in, T* __restrict__ dst, const P3 p,
                        int wb) {
  const int x = blockIdx.x * kBlock3 + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
  if (x >= p.nx) return;
#pragma unroll
  for (int i = 0; i < kQ3; ++i) {
    const int xx = wrap3(x + cx3(i), p.nx), yy = wrap3(y + cy3(i), p.ny),
              zz = wrap3(z + cz3(i), p.nz);
    const size_t from = (size_t)(zz * p.ny + yy) * p.nx + xx;
    const double r = (WB_IN(from, p.nodes) ? rho_in[from] : 0.0) - p.rho_ref;
    // WB: f_0^eq - s_0 = rho - rho_ref, f_i^eq - s_i = 0; standard: w_i (rho - rho_ref)
    const long long k = at3(p, x, y, z);
    if (WB_IN(k, p.plane)) dst[i * p.plane + k] = (T)(wb ? (i == 0 ? r : 0.0) : w3(i) * r);
  }
}

// f_i(x) = P_i(x - c_i) + s_i for one direction, [nz][ny][nx].
template <typename T>
__global__ void d3_get(const T* __restrict__ src, double* __restrict__ f, const P3 p, int dir,
                       double shift) {
  const int x = blockIdx.x * kBlock3 + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
  if (x >= p.nx) return;
  const long long k = at3(p, wrap3(x - cx3(dir), p.nx), wrap3(y - cy3(dir), p.ny),
                          wrap3(z - cz3(dir), p.nz));
  const double v = WB_IN(k, p.plane) ? (double)src[dir * p.plane + k] : 0.0;
  const size_t to = (size_t)(z * p.ny + y) * p.nx + x;
  if (WB_IN(to, p.nodes)) f[to] = v + shift;
}

thread_local char g_d3_error[256] = "";

size_t align3(size_t v) { return (v + kAlign3 - 1) / kAlign3 * kAlign3; }

struct Layout3 {
  int pitch;
  long long plane;
  size_t off_a, off_b, off_rho, off_mu, off_stage, off_partials, off_stats, total;
  int planes;                     // planes per CTA of the moments pass
  long long records;              // its CTAs
};

size_t elem3(const wblbe3_params* p) { return p->precision == WBLBE_FP64 ? 8 : 4; }

Layout3 layout3(const wblbe3_params* p) {
  Layout3 L{};
  L.pitch = (p->nx + 15) / 16 * 16;
  L.plane = (long long)L.pitch * p->ny * p->nz;
  const size_t pops = align3((size_t)kQ3 * L.plane * elem3(p));
  const size_t field = align3((size_t)L.plane * elem3(p));
  // up to 8, while that leaves 400 CTAs (2.6 per SM): with fewer, a CTA's planes
  // one after another are the pass.  us of the whole call with 1, 2, 4 and 8
  // planes: FP64 8^3 42, 42, 50, 58; 32^3 55, 53, 53, 58; 40^3 78, 68, 59, 65; 64^3
  // 131, 109, 105, 101; FP32 24^3 41, 40, 43, 53; 48^3 54, 45, 44, 54; 96^3 123, 97,
  // 82, 79
  const long long rows = (long long)((p->nx + kBlock3 - 1) / kBlock3) * p->ny;
  for (L.planes = 8; L.planes > 1 && rows * ((p->nz + L.planes - 1) / L.planes) < 400;) L.planes /= 2;
  L.records = rows * ((p->nz + L.planes - 1) / L.planes);
  size_t off = 0;
  L.off_a = off; off += pops;
  L.off_b = off; off += pops;
  L.off_rho = off; off += field;
  L.off_mu = off; off += field;
  L.off_stage = off; off += align3((size_t)p->nx * p->ny * p->nz * sizeof(double));
  L.off_partials = off; off += align3((size_t)L.records * kStatRec * sizeof(double));
  L.off_stats = off; off += align3(8 * sizeof(double));
  L.total = off;
  return L;
}

bool params3_valid(const wblbe3_params* p, char* why, size_t n) {
  if (!p) { snprintf(why, n, "params is NULL"); return false; }
  if (p->nx < 1 || p->ny < 1 || p->nz < 1) { snprintf(why, n, "nx, ny, nz must be >= 1"); return false; }
  if (!(p->tau > 0.5) || !std::isfinite(p->tau)) { snprintf(why, n, "tau must be > 0.5"); return false; }
  if (!(p->kappa >= 0.0) || !(p->beta > 0.0)) { snprintf(why, n, "need kappa >= 0, beta > 0"); return false; }
  if (!(p->rho_g > 0.0) || !(p->rho_l > p->rho_g)) { snprintf(why, n, "need rho_l > rho_g > 0"); return false; }
  if (!std::isfinite(p->rho0)) { snprintf(why, n, "rho0 must be finite"); return false; }
  if (p->scheme != WBLBE_STANDARD && p->scheme != WBLBE_WELL_BALANCED) {
    snprintf(why, n, "the D3Q19 path runs the standard and well-balanced schemes"); return false;
  }
  if (p->precision != WBLBE_FP64 && p->precision != WBLBE_FP32_SHIFTED) {
    snprintf(why, n, "unknown precision %d", p->precision); return false;
  }
  // the kernels' element offsets within a plane, and the node numbers of the
  // last block, are 32 bits (Nbr3, node_of)
  if (p->ny > 65535 || p->nz > 65535 || p->nx > INT32_MAX - 15 ||
      (long long)((p->nx + 15) / 16 * 16) * p->ny > kMaxPlane3 / p->nz) {
    snprintf(why, n, "lattice too large (ny, nz <= 65535, fewer than 2^32 elements in a plane)");
    return false;
  }
  return true;
}

// Planes per CTA of the FP32 step kernel: the run whose waves of resident CTAs
// (on nsm SMs) take the fewest plane iterations in all (a run of n planes takes
// n + 4, of which the first four store nothing).
int step_run(const wblbe3_params* p, int nsm) {
  const long long tiles = (long long)((p->nx + kTX3 - 1) / kTX3) * ((p->ny + kTY3 - 1) / kTY3);
  const long long resident = (long long)nsm * kMinB3;
  int best = p->nz;
  long long cost = -1;
  for (int segs = 1; segs <= p->nz && segs <= 65535; ++segs) {
    const int run = (p->nz + segs - 1) / segs;
    const long long n = tiles * ((p->nz + run - 1) / run);
    const long long c = (n + resident - 1) / resident * (run + 4);
    if (cost < 0 || c < cost) {
      cost = c;
      best = run;
    }
  }
  return best;
}

}  // namespace

struct wblbe3_ctx {
  wblbe3_params p;
  Layout3 L;
  int run;                        // planes per CTA of the FP32 step (step_run)
  int device;
  cudaStream_t stream;
  void* buf[2];                   // population buffers (float64 or float32)
  int cur;
  void *rho, *mu;                 // rho - rho_ref and mu fields (the same type)
  double *stage, *partials, *stats;
  int64_t steps, launches;
  double mass0;
  bool have_state;
  char err[256];
};

namespace {

wblbe_status f3(wblbe3_ctx* h, wblbe_status st, const char* fmt, ...) {
  char* dst = h ? h->err : g_d3_error;
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(dst, 256, fmt, ap);
  va_end(ap);
  return st;
}

#define CU3(h, call)                                                         \
  do {                                                                       \
    cudaError_t e_ = (call);                                                 \
    if (e_ != cudaSuccess)                                                   \
      return f3((h), WBLBE_ECUDA, "%s: %s", #call, cudaGetErrorString(e_));  \
  } while (0)

P3 p3_of(const wblbe3_ctx* h) {
  P3 q{};
  q.nx = h->p.nx;
  q.ny = h->p.ny;
  q.nz = h->p.nz;
  q.nodes = (unsigned)((long long)q.nx * q.ny * q.nz);
  q.pitch = h->L.pitch;
  q.plane = h->L.plane;
  // FP32 stores deviations from the rest equilibrium at rho_ref = rho_g
  q.rho_ref = h->p.precision == WBLBE_FP64 ? 0.0 : h->p.rho_g;
  const double om = 1.0 / h->p.tau, kf = 1.0 - 1.0 / (2.0 * h->p.tau), tb = 2.0 * h->p.beta;
  const double dl = q.rho_ref - h->p.rho_l, dg = q.rho_ref - h->p.rho_g;
  q.d.set(om, kf, h->p.kappa, tb, dl, dg, q.rho_ref);
  q.f.set(om, kf, h->p.kappa, tb, dl, dg, q.rho_ref);
  q.kc72 = -kf / 72.0;
  q.kf288 = kf / 288.0;
  q.step = h->steps;
  return q;
}

dim3 grid3(const wblbe3_ctx* h) {
  return dim3((h->p.nx + kBlock3 - 1) / kBlock3, h->p.ny, h->p.nz);
}

// The stored shift s_i: the well-balanced rho0 vector, plus in FP32 the
// scheme's rest equilibrium at rho_ref = rho_g.
double shift3(const wblbe3_params& p, int i) {
  const double rr = p.precision == WBLBE_FP64 ? 0.0 : p.rho_g;
  if (p.scheme != WBLBE_WELL_BALANCED) return w3(i) * rr;
  return i == 0 ? rr - (1.0 - w3(0)) * p.rho0 : w3(i) * p.rho0;
}

// A kernel chained to the stream's previous one (see ChainedLaunch).
template <typename... K, typename... A>
cudaError_t launch3(void (*kernel)(K...), dim3 grid, int block, cudaStream_t s, A... args) {
  ChainedLaunch l(grid, block, 0, s, true);
  return cudaLaunchKernelEx(&l.cfg, kernel, static_cast<K>(args)...);
}

// g: the grid of rows of blocks
template <typename T>
cudaError_t launch_density(cudaStream_t s, const T* src, T* rho, const P3& q, dim3 g) {
  return q.nx % kBlock3 != 0
             ? launch3(d3_density<T, true>, dim3((q.nodes + (unsigned)kBlock3 - 1) / kBlock3),
                       kBlock3, s, src, rho, q)
             : launch3(d3_density<T, false>, g, kBlock3, s, src, rho, q);
}

// Density and chemical potential of the current state, then the moments
// (fields and statistics), or in FP64 the collision into the other buffer.
template <typename T, bool WB>
cudaError_t pass3_typed(wblbe3_ctx* h, bool moments, const Out3& out, const P3& q, dim3 g) {
  const T* src = static_cast<const T*>(h->buf[h->cur]);
  T* rho = static_cast<T*>(h->rho);
  T* mu = static_cast<T*>(h->mu);
  // rows that are whole blocks, or one run of nodes (node_of)
  const bool flat = q.nx % kBlock3 != 0;
  const dim3 gn = flat ? dim3((q.nodes + (unsigned)kBlock3 - 1) / kBlock3) : g;
  cudaError_t e = launch_density(h->stream, src, rho, q, g);
  if (e == cudaSuccess)
    e = flat ? launch3(d3_chem_pot<T, true>, gn, kBlock3, h->stream, rho, mu, q)
             : launch3(d3_chem_pot<T, false>, gn, kBlock3, h->stream, rho, mu, q);
  if (e != cudaSuccess) return e;
  if (moments) {
    const dim3 gm(g.x, g.y, (h->p.nz + h->L.planes - 1) / h->L.planes);
    return launch3(d3_moments<T, WB>, gm, kBlock3, h->stream, src, rho, mu, q, out, h->L.planes);
  }
  if constexpr (sizeof(T) == 8)
    return flat ? launch3(d3_collide<WB, true>, gn, kBlock3, h->stream, src,
                          static_cast<T*>(h->buf[1 - h->cur]), rho, mu, q)
                : launch3(d3_collide<WB, false>, gn, kBlock3, h->stream, src,
                          static_cast<T*>(h->buf[1 - h->cur]), rho, mu, q);
  return cudaErrorInvalidValue;              // FP32 steps: fp32_step
}

cudaError_t fp32_step(wblbe3_ctx* h, const P3& q) {
  const int run = h->run;
  const dim3 grid((h->p.nx + kTX3 - 1) / kTX3, (h->p.ny + kTY3 - 1) / kTY3,
                  (h->p.nz + run - 1) / run);
  const float* src = static_cast<const float*>(h->buf[h->cur]);
  float* dst = static_cast<float*>(h->buf[1 - h->cur]);
  float* rho = static_cast<float*>(h->rho);
  const cudaError_t e = launch_density(h->stream, src, rho, q, grid3(h));
  if (e != cudaSuccess) return e;
  return h->p.scheme == WBLBE_WELL_BALANCED
             ? launch3(d3_step_f32<true>, grid, kNT3, h->stream, src, dst, rho, q, run)
             : launch3(d3_step_f32<false>, grid, kNT3, h->stream, src, dst, rho, q, run);
}

wblbe_status pass3(wblbe3_ctx* h, bool moments, const Out3& out) {
  const P3 q = p3_of(h);
  if (!moments && h->p.precision == WBLBE_FP32_SHIFTED) {
    CU3(h, fp32_step(h, q));
    h->launches += 2;
    return WBLBE_OK;
  }
  const dim3 g = grid3(h);
  const bool wb = h->p.scheme == WBLBE_WELL_BALANCED;
  CU3(h, h->p.precision == WBLBE_FP64
             ? (wb ? pass3_typed<double, true>(h, moments, out, q, g)
                   : pass3_typed<double, false>(h, moments, out, q, g))
             : (wb ? pass3_typed<float, true>(h, moments, out, q, g)
                   : pass3_typed<float, false>(h, moments, out, q, g)));
  h->launches += 3;
  return WBLBE_OK;
}

wblbe_status stats3(wblbe3_ctx* h, double* rho, double* ux, double* uy, double* uz, double* mu,
                    wblbe_stats* st) {
  Out3 out{rho, ux, uy, uz, mu, h->partials};
  wblbe_status s = pass3(h, true, out);
  if (s != WBLBE_OK) return s;
  stats_finalize_kernel<<<1, 256, 0, h->stream>>>(h->partials, (int)h->L.records, h->stats);
  CU3(h, cudaGetLastError());
  h->launches += 1;
  double v[kStatRec];
  CU3(h, cudaMemcpyAsync(v, h->stats, sizeof(v), cudaMemcpyDeviceToHost, h->stream));
  CU3(h, cudaStreamSynchronize(h->stream));
  if (st) {
    st->step = h->steps;
    st->mass = v[0];
    st->kinetic = v[1];
    st->umax = v[2];
    st->mu_min = v[3];
    st->mu_max = v[4];
    st->nonfinite = v[5] != 0.0 || !std::isfinite(v[0]);
    st->mass_drift_rel = h->mass0 != 0.0 ? (v[0] - h->mass0) / h->mass0 : 0.0;
  }
  return WBLBE_OK;
}

}  // namespace

extern "C" {

size_t wblbe3_workspace_bytes(const wblbe3_params* params) {
  char why[256];
  if (!params3_valid(params, why, sizeof(why))) return 0;
  return layout3(params).total;
}

wblbe_status wblbe3_create(const wblbe3_params* params, void* dev_workspace,
                           size_t workspace_bytes, void* cuda_stream, wblbe3_handle* out) {
  char why[256];
  if (!out) return f3(nullptr, WBLBE_EINVAL, "out is NULL");
  *out = nullptr;
  if (!params3_valid(params, why, sizeof(why))) return f3(nullptr, WBLBE_EINVAL, "%s", why);
  const Layout3 L = layout3(params);
  if (!dev_workspace || ((uintptr_t)dev_workspace % kAlign3) != 0)
    return f3(nullptr, WBLBE_EINVAL, "workspace must be a 256-byte aligned device pointer");
  if (workspace_bytes < L.total)
    return f3(nullptr, WBLBE_ENOMEM, "workspace has %zu bytes, needs %zu", workspace_bytes, L.total);
  if (L.records > 0x7fffffffLL) return f3(nullptr, WBLBE_EINVAL, "lattice too large");
  wblbe3_ctx* h = new (std::nothrow) wblbe3_ctx();
  if (!h) return f3(nullptr, WBLBE_ENOMEM, "host allocation failed");
  if (cudaGetDevice(&h->device) != cudaSuccess) {
    delete h;
    return f3(nullptr, WBLBE_ECUDA, "no CUDA device");
  }
  int nsm = 0;
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, h->device) != cudaSuccess ||
      nsm < 1) {
    delete h;
    return f3(nullptr, WBLBE_ECUDA, "cudaDeviceGetAttribute failed");
  }
  unsigned char* ws = static_cast<unsigned char*>(dev_workspace);
  h->p = *params;
  h->L = L;
  h->run = step_run(params, nsm);
  h->stream = static_cast<cudaStream_t>(cuda_stream);
  h->buf[0] = ws + L.off_a;
  h->buf[1] = ws + L.off_b;
  h->rho = ws + L.off_rho;
  h->mu = ws + L.off_mu;
  h->stage = reinterpret_cast<double*>(ws + L.off_stage);
  h->partials = reinterpret_cast<double*>(ws + L.off_partials);
  h->stats = reinterpret_cast<double*>(ws + L.off_stats);
  *out = h;
  return WBLBE_OK;
}

wblbe_status wblbe3_init_rho(wblbe3_handle h, const double* rho, int32_t rho_on_device) {
  if (!h) return f3(nullptr, WBLBE_EINVAL, "handle is NULL");
  if (!rho) return f3(h, WBLBE_EINVAL, "rho is NULL");
  const double* src = rho;
  if (!rho_on_device) {
    CU3(h, cudaMemcpyAsync(h->stage, rho, (size_t)h->p.nx * h->p.ny * h->p.nz * sizeof(double),
                           cudaMemcpyHostToDevice, h->stream));
    src = h->stage;
  }
  h->cur = 0;
  const int wb = h->p.scheme == WBLBE_WELL_BALANCED;
  if (h->p.precision == WBLBE_FP64)
    d3_init<double><<<grid3(h), kBlock3, 0, h->stream>>>(
        src, static_cast<double*>(h->buf[0]), p3_of(h), wb);
  else
    d3_init<float><<<grid3(h), kBlock3, 0, h->stream>>>(
        src, static_cast<float*>(h->buf[0]), p3_of(h), wb);
  CU3(h, cudaGetLastError());
  h->launches += 1;
  h->steps = 0;
  h->have_state = true;
  wblbe_stats s{};
  wblbe_status st = stats3(h, nullptr, nullptr, nullptr, nullptr, nullptr, &s);
  if (st != WBLBE_OK) return st;
  h->mass0 = s.mass;
  return WBLBE_OK;
}

wblbe_status wblbe3_step(wblbe3_handle h, int64_t nsteps) {
  if (!h) return f3(nullptr, WBLBE_EINVAL, "handle is NULL");
  if (nsteps < 0) return f3(h, WBLBE_EINVAL, "nsteps must be >= 0");
  if (!h->have_state) return f3(h, WBLBE_EINVAL, "no state: call wblbe3_init_rho first");
  for (int64_t n = 0; n < nsteps; ++n) {
    wblbe_status st = pass3(h, false, Out3{});
    if (st != WBLBE_OK) return st;
    h->cur ^= 1;
    h->steps += 1;
  }
  return WBLBE_OK;
}

wblbe_status wblbe3_moments(wblbe3_handle h, double* rho, double* u, double* mu,
                            int32_t out_on_device, wblbe_stats* stats) {
  if (!h) return f3(nullptr, WBLBE_EINVAL, "handle is NULL");
  if (!h->have_state) return f3(h, WBLBE_EINVAL, "no state: call wblbe3_init_rho first");
  const size_t n = (size_t)h->p.nx * h->p.ny * h->p.nz;
  if (out_on_device)
    return stats3(h, rho, u, u ? u + n : nullptr, u ? u + 2 * n : nullptr, mu, stats);
  // host outputs: one field at a time through the staging field
  double* outs[5] = {rho, u, u ? u + n : nullptr, u ? u + 2 * n : nullptr, mu};
  bool any = false;
  for (int q = 0; q < 5; ++q) {
    if (!outs[q]) continue;
    any = true;
    double* dev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    dev[q] = h->stage;
    wblbe_status st = stats3(h, dev[0], dev[1], dev[2], dev[3], dev[4], stats);
    if (st != WBLBE_OK) return st;
    CU3(h, cudaMemcpyAsync(outs[q], h->stage, n * sizeof(double), cudaMemcpyDeviceToHost,
                           h->stream));
  }
  if (!any) return stats3(h, nullptr, nullptr, nullptr, nullptr, nullptr, stats);
  CU3(h, cudaStreamSynchronize(h->stream));
  return WBLBE_OK;
}

wblbe_status wblbe3_get_populations(wblbe3_handle h, double* f, int32_t on_device) {
  if (!h) return f3(nullptr, WBLBE_EINVAL, "handle is NULL");
  if (!f) return f3(h, WBLBE_EINVAL, "f is NULL");
  if (!h->have_state) return f3(h, WBLBE_EINVAL, "no state: call wblbe3_init_rho first");
  const size_t n = (size_t)h->p.nx * h->p.ny * h->p.nz;
  for (int i = 0; i < kQ3; ++i) {
    double* dst = on_device ? f + i * n : h->stage;
    if (h->p.precision == WBLBE_FP64)
      d3_get<double><<<grid3(h), kBlock3, 0, h->stream>>>(
          static_cast<const double*>(h->buf[h->cur]), dst, p3_of(h), i, shift3(h->p, i));
    else
      d3_get<float><<<grid3(h), kBlock3, 0, h->stream>>>(
          static_cast<const float*>(h->buf[h->cur]), dst, p3_of(h), i, shift3(h->p, i));
    CU3(h, cudaGetLastError());
    h->launches += 1;
    if (!on_device)
      CU3(h, cudaMemcpyAsync(f + i * n, h->stage, n * sizeof(double), cudaMemcpyDeviceToHost,
                             h->stream));
  }
  CU3(h, cudaStreamSynchronize(h->stream));
  return WBLBE_OK;
}

int64_t wblbe3_step_count(wblbe3_handle h) { return h ? h->steps : -1; }
int64_t wblbe3_kernel_launches(wblbe3_handle h) { return h ? h->launches : -1; }

wblbe_status wblbe3_destroy(wblbe3_handle h) {
  if (!h) return f3(nullptr, WBLBE_EINVAL, "handle is NULL");
  cudaStreamSynchronize(h->stream);
  delete h;
  return WBLBE_OK;
}

const char* wblbe3_last_error(wblbe3_handle h) { return h ? h->err : g_d3_error; }

}  // extern "C"

namespace wblbe {
// bounds-check count of this translation unit's kernels (see lbm_kernels.cuh)
unsigned int d3_bounds_errors(bool reset) { return read_bounds_errors(reset); }
}  // namespace wblbe
