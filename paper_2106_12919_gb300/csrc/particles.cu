// Particle stage of the hybrid cycle (Sec. 2): gather E, B from the nodal grid
// with B-spline shapes, Boris push, move, direct deposition of J^{n+1/2} and
// rho^{n+1} on the nodal grid; and tile binning of the particle SoA.
//
// Shapes (textbook centred B-splines on the nodal grid, node i at i dx):
//   order 1: base = floor(t), d = t - base; nodes base..base+1
//   order 2: base = floor(t + 1/2);          nodes base-1..base+1
//   order 3: base = floor(t);                nodes base-1..base+2
// with t = x * (1/dx) as one correctly rounded multiply (__dmul_rn) so that the
// integer cell decision is the same on every implementation.
// Node indices wrap with & (N - 1) (N a power of two), which also keeps every
// access in bounds whatever the position value.
#include "pic_internal.cuh"

#include <algorithm>

namespace {

struct PushArgs {
  double *x, *y, *z, *ux, *uy, *uz;
  const double* w;
  int64_t n;
  const double* F[6];  // nodal Ex, Ey, Ez, Bx, By, Bz
  double* J[3];        // nodal J deposit (atomic add)
  double* rho;         // nodal rho deposit (atomic add)
  double inv_dx[3];
  double L[3];
  int mask[3];
  int64_t Ny, Nz;
  double qm_half_dt;   // q dt / (2 m)
  double dt;
  double inv_c2;
  double vg[3];
  double qw_scale;     // q / dV
  int gather;          // 0: rho-only deposit at the current position
  int vay;             // 1: Vay's pusher instead of Boris
};

// shape of order P at position x on a grid whose points sit at (i + off) dx (off = 0: nodes,
// off = 1/2: a staggered Yee axis): t = x / dx - off
template <int P>
__device__ __forceinline__ void shape(double x, double inv, int mask, int& lo, double* S, double off = 0.0) {
  const double t = __dmul_rn(x, inv) - off;
  int b;
  const double d = t - floor_cell(P == 2 ? __dadd_rn(t, 0.5) : t, b);
  if (P == 1) {
    lo = b;
    S[0] = 1.0 - d;
    S[1] = d;
  } else if (P == 2) {
    lo = b - 1;
    const double a = 0.5 - d, c = 0.5 + d;
    S[0] = 0.5 * a * a;
    S[1] = 0.75 - d * d;
    S[2] = 0.5 * c * c;
  } else {
    lo = b - 1;
    // the inner weights as 2/3 + d^2 (d/2 - 1) and its mirror image
    const double e = 1.0 - d, d2 = d * d, e2 = e * e;
    S[0] = e2 * (e * (1.0 / 6.0));
    S[1] = fma(d2, fma(0.5, d, -1.0), 2.0 / 3.0);
    S[2] = fma(e2, fma(0.5, e, -1.0), 2.0 / 3.0);
    S[3] = d2 * (d * (1.0 / 6.0));
  }
  (void)mask;
}

// u^{n-1/2} of particle p -> u^{n+1/2} with the gathered f = (E, B): Boris rotation, or Vay's pusher
__device__ __forceinline__ void push_u(const PushArgs& a, int64_t p, const double* f, double& ux, double& uy,
                                       double& uz) {
  const double k = a.qm_half_dt;
  if (a.vay) {
    ux = a.ux[p];
    uy = a.uy[p];
    uz = a.uz[p];
    vay_push<double>(ux, uy, uz, f, k, a.inv_c2);
    return;
  }
  const double umx = a.ux[p] + k * f[0], umy = a.uy[p] + k * f[1], umz = a.uz[p] + k * f[2];
  // (one rsqrt instead of a square root and three divisions: FP64 divisions cost about ten operations)
  const double igm = rsqrt(1.0 + (umx * umx + umy * umy + umz * umz) * a.inv_c2);
  const double tx = k * f[3] * igm, ty = k * f[4] * igm, tz = k * f[5] * igm;
  const double s2 = 2.0 / (1.0 + tx * tx + ty * ty + tz * tz);
  const double sx = s2 * tx, sy = s2 * ty, sz = s2 * tz;
  const double upx = fma(umy, tz, fma(-umz, ty, umx));
  const double upy = fma(umz, tx, fma(-umx, tz, umy));
  const double upz = fma(umx, ty, fma(-umy, tx, umz));
  ux = fma(upy, sz, fma(-upz, sy, fma(k, f[0], umx)));
  uy = fma(upz, sx, fma(-upx, sz, fma(k, f[1], umy)));
  uz = fma(upx, sy, fma(-upy, sx, fma(k, f[2], umz)));
}

// x in [0, L) after a move of less than a period; the comparisons are on the bit patterns (of positive
// doubles, ordered as integers), off the FP64 pipe
__device__ __forceinline__ double wrap(double x, double L) {
  if (__double_as_longlong(x) >= __double_as_longlong(L)) x -= L;  // x >= L > 0 (or not finite)
  if (__double_as_longlong(x) < 0 && x < 0.0) x += L;
  return x;
}

// rho of one particle: node (i, j, k) receives (Sx_i q w)(Sy_j Sz_k); Syz is the caller's storage
template <int P>
__device__ __forceinline__ void deposit_rho_nodes(const PushArgs& a, int lx, int ly, int lz, const double* Sx,
                                                  const double* Sy, const double* Sz, double qw,
                                                  double (&Syz)[P + 1][P + 1]) {
  constexpr int NS = P + 1;
  double Sq[NS];
#pragma unroll
  for (int i = 0; i < NS; ++i) Sq[i] = Sx[i] * qw;
#pragma unroll
  for (int j = 0; j < NS; ++j)
#pragma unroll
    for (int k = 0; k < NS; ++k) Syz[j][k] = Sy[j] * Sz[k];
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const int64_t ox = (int64_t)((lx + i) & a.mask[0]) * a.Ny;
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      const int64_t oy = (ox + ((ly + j) & a.mask[1])) * a.Nz;
#pragma unroll
      for (int k = 0; k < NS; ++k) atomicAdd(a.rho + oy + ((lz + k) & a.mask[2]), Sq[i] * Syz[j][k]);
    }
  }
}

template <int P>
__device__ __forceinline__ void push_particle(const PushArgs& a, int64_t p) {
  constexpr int NS = P + 1;
  const double x = a.x[p], y = a.y[p], z = a.z[p];
  const double qw = a.w[p] * a.qw_scale;
  int lx, ly, lz;
  double Sx[NS], Sy[NS], Sz[NS];
  // The weight of node (i, j, k) is Sx_i Sy_j Sz_k.  Every sum below forms the NS^2 products
  // Sy_j Sz_k once and carries the particle's factor (q w, or q w v_c) on the NS x weights, so a
  // node costs one FP64 multiply or FMA per value instead of two (the FP64 pipe bounds this kernel).
  double Syz[NS][NS];
  if (!a.gather) {
    shape<P>(x, a.inv_dx[0], a.mask[0], lx, Sx);
    shape<P>(y, a.inv_dx[1], a.mask[1], ly, Sy);
    shape<P>(z, a.inv_dx[2], a.mask[2], lz, Sz);
    deposit_rho_nodes<P>(a, lx, ly, lz, Sx, Sy, Sz, qw, Syz);
    return;
  }
  shape<P>(x, a.inv_dx[0], a.mask[0], lx, Sx);
  shape<P>(y, a.inv_dx[1], a.mask[1], ly, Sy);
  shape<P>(z, a.inv_dx[2], a.mask[2], lz, Sz);
  // gather E, B at x^n: f_c = sum_i Sx_i g_ic, g_ic = sum_jk (Sy_j Sz_k) F_c(i, j, k)
#pragma unroll
  for (int j = 0; j < NS; ++j)
#pragma unroll
    for (int k = 0; k < NS; ++k) Syz[j][k] = Sy[j] * Sz[k];
  double f[6];
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const int64_t ox = (int64_t)((lx + i) & a.mask[0]) * a.Ny;
    double g[6];
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      const int64_t oy = (ox + ((ly + j) & a.mask[1])) * a.Nz;
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        const int64_t o = oy + ((lz + k) & a.mask[2]);
#pragma unroll
        for (int c = 0; c < 6; ++c) {
          const double v = __ldg(a.F[c] + o);
          g[c] = (j == 0 && k == 0) ? Syz[j][k] * v : fma(Syz[j][k], v, g[c]);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) f[c] = i == 0 ? Sx[0] * g[c] : fma(Sx[i], g[c], f[c]);
  }
  // push u^{n-1/2} -> u^{n+1/2}
  double ux, uy, uz;
  push_u(a, p, f, ux, uy, uz);
  const double ig = rsqrt(1.0 + (ux * ux + uy * uy + uz * uz) * a.inv_c2);
  const double vx = ux * ig, vy = uy * ig, vz = uz * ig;
  // move: x^{n+1} = x^n + dt (v - v_gal); J at x^{n+1/2}
  const double dX = a.dt * (vx - a.vg[0]), dY = a.dt * (vy - a.vg[1]), dZ = a.dt * (vz - a.vg[2]);
  const double mx = wrap(x + 0.5 * dX, a.L[0]), my = wrap(y + 0.5 * dY, a.L[1]), mz = wrap(z + 0.5 * dZ, a.L[2]);
  const double nx = wrap(x + dX, a.L[0]), ny = wrap(y + dY, a.L[1]), nz = wrap(z + dZ, a.L[2]);
  a.x[p] = nx;
  a.y[p] = ny;
  a.z[p] = nz;
  a.ux[p] = ux;
  a.uy[p] = uy;
  a.uz[p] = uz;
  // J^{n+1/2} = q w v S(x^{n+1/2} - x_i) / dV
  shape<P>(mx, a.inv_dx[0], a.mask[0], lx, Sx);
  shape<P>(my, a.inv_dx[1], a.mask[1], ly, Sy);
  shape<P>(mz, a.inv_dx[2], a.mask[2], lz, Sz);
  const double jx = qw * vx, jy = qw * vy, jz = qw * vz;
  double Sj[3][NS];  // (Sx_i q w v_c)
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    Sj[0][i] = Sx[i] * jx;
    Sj[1][i] = Sx[i] * jy;
    Sj[2][i] = Sx[i] * jz;
  }
#pragma unroll
  for (int j = 0; j < NS; ++j)
#pragma unroll
    for (int k = 0; k < NS; ++k) Syz[j][k] = Sy[j] * Sz[k];
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const int64_t ox = (int64_t)((lx + i) & a.mask[0]) * a.Ny;
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      const int64_t oy = (ox + ((ly + j) & a.mask[1])) * a.Nz;
#pragma unroll
      for (int kk = 0; kk < NS; ++kk) {
        const int64_t o = oy + ((lz + kk) & a.mask[2]);
        atomicAdd(a.J[0] + o, Sj[0][i] * Syz[j][kk]);
        atomicAdd(a.J[1] + o, Sj[1][i] * Syz[j][kk]);
        atomicAdd(a.J[2] + o, Sj[2][i] * Syz[j][kk]);
      }
    }
  }
  // rho^{n+1} = q w S(x^{n+1} - x_i) / dV
  shape<P>(nx, a.inv_dx[0], a.mask[0], lx, Sx);
  shape<P>(ny, a.inv_dx[1], a.mask[1], ly, Sy);
  shape<P>(nz, a.inv_dx[2], a.mask[2], lz, Sz);
  deposit_rho_nodes<P>(a, lx, ly, lz, Sx, Sy, Sz, qw, Syz);
}

// The cubic form holds 128 registers (2 CTAs of 256 threads per SM, no spills); orders 1 and 2 keep
// the compiler's own choice (64 and ~100 registers).
template <int P>
__global__ void __launch_bounds__(256) push_kernel(PushArgs a) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p < a.n) push_particle<P>(a, p);
}
template <>
__global__ void __launch_bounds__(256, 2) push_kernel<3>(PushArgs a) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p < a.n) push_particle<3>(a, p);
}

// Staggered comparison cycle (Sec. 2): E, B are gathered from their own Yee positions and J is
// deposited at its Yee positions (rho stays nodal).  Component c is staggered along the axes of
// its bit mask (E: x, y, z; B: yz, xz, xy); shapes on the staggered axes use offset 1/2.
template <int P>
__device__ __forceinline__ double gather_one(const double* F, const PushArgs& a, const int* lo, const double* Sx,
                                             const double* Sy, const double* Sz) {
  constexpr int NS = P + 1;
  double v = 0.0;
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const int64_t ox = (int64_t)((lo[0] + i) & a.mask[0]) * a.Ny;
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      const int64_t oy = (ox + ((lo[1] + j) & a.mask[1])) * a.Nz;
      const double sxy = Sx[i] * Sy[j];
#pragma unroll
      for (int k = 0; k < NS; ++k) v += sxy * Sz[k] * __ldg(F + oy + ((lo[2] + k) & a.mask[2]));
    }
  }
  return v;
}

template <int P>
__device__ __forceinline__ void deposit_one(double* F, const PushArgs& a, const int* lo, const double* Sx,
                                            const double* Sy, const double* Sz, double val) {
  constexpr int NS = P + 1;
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const int64_t ox = (int64_t)((lo[0] + i) & a.mask[0]) * a.Ny;
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      const int64_t oy = (ox + ((lo[1] + j) & a.mask[1])) * a.Nz;
      const double sxy = Sx[i] * Sy[j] * val;
#pragma unroll
      for (int k = 0; k < NS; ++k) atomicAdd(F + oy + ((lo[2] + k) & a.mask[2]), sxy * Sz[k]);
    }
  }
}

template <int P>
__global__ void __launch_bounds__(256) push_stag_kernel(PushArgs a) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= a.n) return;
  constexpr int NS = P + 1;
  const double x[3] = {a.x[p], a.y[p], a.z[p]};
  const double qw = a.w[p] * a.qw_scale;
  // shapes on the nodal (0) and staggered (1) grid of every axis
  int l0[3], l1[3];
  double S0[3][NS], S1[3][NS];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    shape<P>(x[d], a.inv_dx[d], a.mask[d], l0[d], S0[d], 0.0);
    shape<P>(x[d], a.inv_dx[d], a.mask[d], l1[d], S1[d], 0.5);
  }
  constexpr int kStag[6] = {1, 2, 4, 6, 5, 3};  // Ex, Ey, Ez, Bx, By, Bz
  double f[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const int m = kStag[c];
    const int lo[3] = {(m & 1) ? l1[0] : l0[0], (m & 2) ? l1[1] : l0[1], (m & 4) ? l1[2] : l0[2]};
    f[c] = gather_one<P>(a.F[c], a, lo, (m & 1) ? S1[0] : S0[0], (m & 2) ? S1[1] : S0[1], (m & 4) ? S1[2] : S0[2]);
  }
  double ux, uy, uz;
  push_u(a, p, f, ux, uy, uz);
  const double ig = rsqrt(1.0 + (ux * ux + uy * uy + uz * uz) * a.inv_c2);
  const double v[3] = {ux * ig, uy * ig, uz * ig};
  double mid[3], nw[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double dd = a.dt * (v[d] - a.vg[d]);
    mid[d] = wrap(x[d] + 0.5 * dd, a.L[d]);
    nw[d] = wrap(x[d] + dd, a.L[d]);
  }
  a.x[p] = nw[0];
  a.y[p] = nw[1];
  a.z[p] = nw[2];
  a.ux[p] = ux;
  a.uy[p] = uy;
  a.uz[p] = uz;
  // J^{n+1/2}: component d at its Yee positions (staggered along axis d)
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    shape<P>(mid[d], a.inv_dx[d], a.mask[d], l0[d], S0[d], 0.0);
    shape<P>(mid[d], a.inv_dx[d], a.mask[d], l1[d], S1[d], 0.5);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int lo[3] = {c == 0 ? l1[0] : l0[0], c == 1 ? l1[1] : l0[1], c == 2 ? l1[2] : l0[2]};
    deposit_one<P>(a.J[c], a, lo, c == 0 ? S1[0] : S0[0], c == 1 ? S1[1] : S0[1], c == 2 ? S1[2] : S0[2],
                   qw * v[c]);
  }
  // rho^{n+1} on the nodes
#pragma unroll
  for (int d = 0; d < 3; ++d) shape<P>(nw[d], a.inv_dx[d], a.mask[d], l0[d], S0[d], 0.0);
  deposit_one<P>(a.rho, a, l0, S0[0], S0[1], S0[2], qw);
}

// ---------------------------------------------------------------------------
// Tiled FP64 push in integer arithmetic.
//
// The untiled push_kernel is bound by this part's FP64 pipe (1.7 lane-operations per clock per SM,
// 1/64 of the FP32 rate): 728 of the ~1030 FP64 operations of a cubic particle are the sums over
// stencil nodes.  Here those run as 32 x 32 -> 64-bit integer multiply-adds (32 per clock per SM) on
// fixed-point values held in two 28-bit limbs, which carry more bits than a double's 53:
//   - shape weights: fractions of 2^56.  x / dx is one correctly rounded FP64 multiply, as in
//     push_kernel (the same cell); its fraction and the polynomials of it are integer.
//   - the tile's nodal E, B, staged in shared memory: 59-bit integers in units of 2^-58 of the power
//     of two above the component's largest node value in the tile.
//   - the deposit window: 64-bit integers in units that keep every node's sum below 2^63 (node_bounds);
//     two 32-bit shared atomics with the carry passed between them add one contribution (a 64-bit
//     shared atomic runs at 1/6 of their rate).  A particle's amounts q w v and q w are 59-bit integers
//     of these units, or of up to 2^5 of them where the amount alone takes more.
// A product of two such values keeps hi * hi + (hi * lo + lo * hi) / 2^28 (the rest is below one
// unit); the node sums themselves are exact, independent of the order of the atomics.  The Boris or
// Vay push and the move stay in FP64 on unchanged formulas.
//
// The particles are not moved: every push first lists the particle numbers by tile (tile64_*_kernel),
// so a particle is always in the tile that stages its nodes, and the library's own tile binning (its
// order, its interval) is as before.  A particle the integers do not cover goes through push_particle
// on its own (global gathers and atomics): a non-finite value or one outside the grid, one that moves
// past the window (over a cell in a step), a chunk whose nodes hold non-finite or vanishing (< 1e-277)
// fields, a chunk of under kMinTiled particles (staging and flushing a tile costs what they save).
// ---------------------------------------------------------------------------
constexpr int kT64 = 8;                    // tile edge in cells
constexpr int kG64 = kT64 + 3;             // staged nodes [T0 - 1, T0 + 10)
constexpr int kW64 = kT64 + 5;             // deposit window nodes [T0 - 2, T0 + 11)
constexpr int kG64n = kG64 * kG64 * kG64;
constexpr int kW64n = kW64 * kW64 * kW64;
// particles per CTA: at most kChunk64, fewer where that leaves SMs without a chunk (chunk64)
constexpr int kChunk64 = 2048, kChunk64Min = 256;
// 2 CTAs of 512 threads per SM, at 64 registers with ~0.9 KB of spills per thread: measured on 4 steps of
// 2.1 million cubic particles, push 5.47 ms; 3 CTAs of 256 at 80 registers 5.62, of 192 at 96 6.6, of 128
// at 168 (no spills) 6.7, 2 of 256 at 128 6.1: no pipe is busy over half of the time, so warps count most
constexpr int kThreads64 = 512;
constexpr int kMinTiled = 16;
// rho by itself (pic_deposit_rho) from this many particles: 131072 cubic ones take 53 us this way and 55 one
// by one (bound by the FP64 pipe: 120 operations each), 1.06 million 189 and 294, 2.1 million 277 and 539
constexpr int64_t kMinRho64 = 1 << 18;
constexpr int kB64 = kW64 - 2;             // first nodes of shape blocks in the window (node_bounds)
constexpr int kB64n = kB64 * kB64 * kB64;
constexpr size_t kWin64 = (size_t)kW64n * 4 * 8;   // >= the staged fields, kG64n * 48
constexpr size_t kSmem64 = kWin64 + (size_t)4 * kB64n * sizeof(float);
constexpr int64_t kMask28 = (int64_t(1) << 28) - 1;
static_assert(kWin64 >= (size_t)kG64n * 48, "the fields and the window share the memory");

struct Tile64Args {
  const int32_t* idx;     // particle numbers grouped by tile
  const int32_t* off;     // [n_tiles + 1] ranges of idx
  const int32_t* cstart;  // [n_tiles + 1] chunks before each tile
  const int32_t* ctile;   // tile of each chunk
  int n_tiles;
  int nt[3];
  int64_t* stash;         // [10][cap]: midpoint, new position (x, y, z each), q w v (3), q w
  int64_t cap;
};

// a fraction of 2^56 (or a signed value) in two limbs: value = h 2^28 + l, 0 <= l < 2^28
struct Limb {
  int h, l;
};
__device__ __forceinline__ Limb limbs(int64_t v) { return {(int)(v >> 28), (int)(v & kMask28)}; }
// a b + c.  In PTX: where the compiler knows one factor's sign and not the other's it forms a full
// 64 x 64-bit product instead (17400 instead of 11500 instructions per cubic particle)
__device__ __forceinline__ int64_t mad_wide(int a, int b, int64_t c) {
  int64_t d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}
// a b / 2^56, rounded
__device__ __forceinline__ int64_t mul56(Limb a, Limb b) {
  return mad_wide(a.h, b.h, mad_wide(a.h, b.l, mad_wide(a.l, b.h, int64_t(1) << 27)) >> 28);
}

// |v| in units of 2^(ref - 1080), rounded, with v's sign: below 2^58 for every v whose biased exponent
// is at most ref
__device__ __forceinline__ int64_t to_fixed58(double v, int ref) {
  const int64_t b = __double_as_longlong(v);
  const int e = (int)(b >> 52) & 0x7ff;
  const int64_t m = ((b & ((int64_t(1) << 52) - 1)) | (e ? int64_t(1) << 52 : 0)) << 5;
  const int sh = ref - max(e, 1);
  const int64_t f = sh < 60 ? (m + ((int64_t(1) << sh) >> 1)) >> sh : 0;
  return b < 0 ? -f : f;
}
// v 2^ex rounded to nearest (half away from zero); the result is a normal double for the ranges used
__device__ __forceinline__ double from_fixed(int64_t v, int ex) {
  if (v == 0) return 0.0;
  const uint64_t a = v < 0 ? (uint64_t)-v : (uint64_t)v;
  const int lz = __clzll((long long)a);
  const uint64_t m = a << lz;
  const uint64_t r = (m >> 11) + ((m >> 10) & 1);  // 53 bits, the leading one adds 1 to the exponent
  const uint64_t bits = ((uint64_t)(1023 + 63 - lz + ex - 1) << 52) + r;
  return __longlong_as_double((int64_t)(bits | (v < 0 ? uint64_t(1) << 63 : 0)));
}

// weights (fractions of 2^56) of order P for the 56-bit fraction d: of x / dx (orders 1, 3) or of
// x / dx + 1/2 (order 2)
template <int P>
__device__ __forceinline__ void weights56(int64_t d, int64_t* S) {
  constexpr int64_t one = int64_t(1) << 56;
  if (P == 2) {
    const Limb a = limbs(one - d), c = limbs(d);
    S[0] = mul56(a, a) >> 1;
    S[2] = mul56(c, c) >> 1;
    S[1] = one - S[0] - S[2];
  } else {
    // (the differences cancel, but in units of 2^-56 that costs one or two units)
    constexpr int64_t sixth = (one + 3) / 6;
    const Limb ld = limbs(d);
    const int64_t d2 = mul56(ld, ld), d3 = mul56(limbs(d2), ld);
    S[3] = mul56(limbs(d3), limbs(sixth));
    S[0] = sixth - ((d - d2) >> 1) - S[3];
    S[1] = 4 * sixth - d2 + (d3 >> 1);
    S[2] = one - S[0] - S[1] - S[3];
  }
}

// x / dx = cell + fraction of 2^56, from the correctly rounded product (bits below 2^-52 of a cell are
// dropped: less than the product's own rounding everywhere but in the first cells); order 2 adds 1/2
// first (its base is the nearest node).  false: negative, beyond 2^10 cells or not finite
template <int P>
__device__ __forceinline__ bool split56(double x, double inv, int& base, int64_t& d) {
  const int64_t b = __double_as_longlong(__dmul_rn(x, inv));
  const int e = (int)(b >> 52);  // sign and biased exponent
  if ((unsigned)e > 1023u + 10u) return false;
  const int64_t m = (b & ((int64_t(1) << 52) - 1)) | (e ? int64_t(1) << 52 : 0);
  const int sh = 1023 - e;       // t = m 2^-52-sh
  int64_t t = sh <= 0 ? m << -sh : (sh < 54 ? m >> sh : 0);  // units of 2^-52
  if (P == 2) t += int64_t(1) << 51;
  base = (int)(t >> 52);
  d = (t & ((int64_t(1) << 52) - 1)) << 4;
  return true;
}

template <int P>
__device__ __noinline__ void push_particle_alone(const PushArgs& a, int64_t p) {
  push_particle<P>(a, p);
}

__device__ __forceinline__ bool finite_bits(double v) {
  return ((__double_as_longlong(v) >> 52) & 0x7ff) != 0x7ff;
}
__device__ __forceinline__ int exponent_of(double v) { return (int)(__double_as_longlong(v) >> 52) & 0x7ff; }

__device__ __forceinline__ void window_add(uint32_t* lo, uint32_t* hi, int64_t c) {
  const uint32_t cl = (uint32_t)c;
  const uint32_t sum = atomicAdd(lo, cl) + cl;
  atomicAdd(hi, (uint32_t)(c >> 32) + (sum < cl ? 1u : 0u));
}

// rows of the deposit block: weight limbs of Sx_i Sy_j times the amounts, then times Sz_k, into the
// window.  The amounts are in units of 2^(l + lz) window units: l <= kRowShift goes onto the rows, whose
// high limb it keeps within 32 bits, lz <= 3 onto the weights Sz_k.
template <int P>
constexpr int kRowShift = P == 2 ? 1 : 2;  // 9/16 2^59 and 4/9 2^60 are below 2^59
template <int P, int NC>
__device__ __forceinline__ void deposit56(uint32_t* win, int c0, const int64_t* pos, const int64_t* amount,
                                          const int* l, int lz) {
  constexpr int NS = P + 1;
  int64_t Sx[NS], Sy[NS], Sz[NS];
  int w[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) w[d] = (int)(pos[d] >> 56);
  constexpr int64_t frac = (int64_t(1) << 56) - 1;
  weights56<P>(pos[0] & frac, Sx);
  weights56<P>(pos[1] & frac, Sy);
  weights56<P>(pos[2] & frac, Sz);
  Limb Z[NS], A[NC];
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    Z[k] = limbs(Sz[k]);
    Z[k].h <<= lz;
    Z[k].l <<= lz;
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) A[c] = limbs(amount[c]);
  const int n0 = (w[0] * kW64 + w[1]) * kW64 + w[2];
#pragma unroll 1
  for (int i = 0; i < NS; ++i) {
    const Limb lx = limbs(Sx[i]);
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      const Limb lxy = limbs(mul56(lx, limbs(Sy[j])));
      Limb row[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) row[c] = limbs(mul56(A[c], lxy) << l[c]);
      uint32_t* p = win + n0 + (i * kW64 + j) * kW64;
#pragma unroll
      for (int k = 0; k < NS; ++k)
#pragma unroll
        for (int c = 0; c < NC; ++c)
          window_add(p + (c0 + c) * kW64n + k, p + (4 + c0 + c) * kW64n + k, mul56(row[c], Z[k]));
    }
  }
}

// Upper bounds of the node sums of a chunk's deposits, the largest per component into out.  blk[c][...]
// holds the sums of |amount c| over the particles whose shape block starts at each window node; a node
// takes at most the largest weights (1/6, 2/3, 2/3, 1/6 per axis of a cubic particle, 1/2, 3/4, 1/2 of a
// quadratic one) of those of the blocks that reach it.  The bound decides the sums' unit: from the
// chunk's total times the largest weight it is 30 times larger at 2 particles per cell, and J of random
// momenta came out 5.4e-15 off the exact one; with this 1.8e-15, as with FP64 atomics.
// tmp: 4 kW64 kB64 (kB64 + kW64) floats.  Components C0 .. 3 only.  Called by the whole CTA.
template <int P, int C0>
__device__ __forceinline__ void node_bounds(const float* blk, float* tmp, unsigned* out) {
  // the sum over the slots s of the largest weight in slot s times v[(n - s) * stride], n - s in [0, kB64)
  const auto line = [](const float* v, int n, int stride) {
    float b = 0.0f;
#pragma unroll
    for (int s = 0; s <= P; ++s) {
      const float w = P == 3 ? (s == 0 || s == 3 ? 0.166667f : 0.666667f) : (s == 1 ? 0.75f : 0.5f);
      if (n - s >= 0 && n - s < kB64) b += w * v[(n - s) * stride];
    }
    return b;
  };
  constexpr int B2 = kB64 * kB64;
  float* X = tmp;                    // [4][kW64][kB64][kB64]
  float* Y = tmp + 4 * kW64 * B2;    // [4][kW64][kW64][kB64]
  for (int e = threadIdx.x + C0 * kW64 * B2; e < 4 * kW64 * B2; e += kThreads64) {
    const int yz = e % B2, n = e / B2 % kW64, c = e / B2 / kW64;
    X[e] = line(blk + c * kB64n + yz, n, B2);
  }
  __syncthreads();
  for (int e = threadIdx.x + C0 * kW64 * kW64 * kB64; e < 4 * kW64 * kW64 * kB64; e += kThreads64) {
    const int z = e % kB64, n = e / kB64 % kW64, cx = e / kB64 / kW64;
    Y[e] = line(X + cx * B2 + z, n, kB64);
  }
  __syncthreads();
  for (int c = C0; c < 4; ++c) {
    float mx = 0.0f;
    for (int e = threadIdx.x; e < kW64n; e += kThreads64)
      mx = fmaxf(mx, line(Y + (c * kW64 * kW64 + e / kW64) * kB64, e % kW64, 1));
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));  // >= 0: ordered as integers
    if ((threadIdx.x & 31) == 0) atomicMax(out + c, m);
  }
  __syncthreads();
}
static_assert((size_t)4 * kW64 * kB64 * (kB64 + kW64) * sizeof(float) <= kWin64, "node_bounds");

// RHO: only rho of the particles as they are (no fields, no push, no J; see kMinRho64)
template <int P, bool RHO>
__global__ void __launch_bounds__(kThreads64, 2) push64_tile_kernel(const __grid_constant__ PushArgs a, Tile64Args t) {
  constexpr int NS = P + 1;
  extern __shared__ __align__(16) unsigned char smraw64[];
  __shared__ int s_chunk[3];       // tile, first particle, count
  __shared__ unsigned s_fmax[6];   // largest biased exponent of each field component in the tile
  __shared__ unsigned s_amax[4];   // of |q w v_c| and |q w|
  __shared__ unsigned s_bound[4];  // largest bounds of their node sums
  if (threadIdx.x == 0) {
    const int b = blockIdx.x;
    s_chunk[0] = -1;
    if (b < t.cstart[t.n_tiles]) {
      const int tl = t.ctile[b], k = b - t.cstart[tl], nch = t.cstart[tl + 1] - t.cstart[tl];
      const int64_t b0 = t.off[tl], cnt = t.off[tl + 1] - b0;
      s_chunk[0] = tl;
      s_chunk[1] = (int)(b0 + cnt * k / nch);
      s_chunk[2] = (int)(b0 + cnt * (k + 1) / nch) - s_chunk[1];
    }
  }
  if (threadIdx.x < 6) s_fmax[threadIdx.x] = 0u;
  if (threadIdx.x < 4) {
    s_amax[threadIdx.x] = 0u;
    s_bound[threadIdx.x] = 0u;
  }
  float* s_blk = reinterpret_cast<float*>(smraw64 + kWin64);
  __syncthreads();
  const int tile = s_chunk[0], p0 = s_chunk[1], cnt = s_chunk[2];
  if (tile < 0) return;
  const int T0[3] = {tile / (t.nt[1] * t.nt[2]) * kT64, tile / t.nt[2] % t.nt[1] * kT64, tile % t.nt[2] * kT64};
  const int Ny = (int)a.Ny, Nz = (int)a.Nz;
  bool alone = cnt < kMinTiled;
  for (int e = threadIdx.x; e < 4 * kB64n; e += kThreads64) s_blk[e] = 0.0f;  // (synchronised below)
  // [3][kG64n] pairs of components: first the doubles, then (h, l) limbs of each in their place
  int4* fld = reinterpret_cast<int4*>(smraw64);
  if (!RHO && !alone) {
    unsigned mx[6] = {0u, 0u, 0u, 0u, 0u, 0u};
    for (int e = threadIdx.x; e < kG64n; e += kThreads64) {
      const int k = e % kG64, r = e / kG64, j = r % kG64, i = r / kG64;
      const int o = (((T0[0] - 1 + i) & a.mask[0]) * Ny + ((T0[1] - 1 + j) & a.mask[1])) * Nz + ((T0[2] - 1 + k) & a.mask[2]);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const double2 v = make_double2(__ldg(a.F[2 * q] + o), __ldg(a.F[2 * q + 1] + o));
        reinterpret_cast<double2*>(fld)[q * kG64n + e] = v;
        mx[2 * q] = max(mx[2 * q], (unsigned)exponent_of(v.x));
        mx[2 * q + 1] = max(mx[2 * q + 1], (unsigned)exponent_of(v.y));
      }
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const unsigned m = __reduce_max_sync(0xffffffffu, mx[c]);
      if ((threadIdx.x & 31) == 0) atomicMax(&s_fmax[c], m);
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 6; ++c) alone = alone || s_fmax[c] == 0x7ffu || (s_fmax[c] > 0u && s_fmax[c] < 100u);
  }
  if (alone) {  // uniform over the CTA
    for (int j = threadIdx.x; j < cnt; j += kThreads64) push_particle_alone<P>(a, t.idx[p0 + j]);
    return;
  }
  for (int e = threadIdx.x; !RHO && e < kG64n; e += kThreads64) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const double2 v = reinterpret_cast<double2*>(fld)[q * kG64n + e];
      const Limb x = limbs(to_fixed58(v.x, (int)s_fmax[2 * q])), y = limbs(to_fixed58(v.y, (int)s_fmax[2 * q + 1]));
      fld[q * kG64n + e] = make_int4(x.h, x.l, y.h, y.l);
    }
  }
  __syncthreads();
  // visit every s-th particle of the list, s ~ the chunk's particles per cell: neighbouring lanes then
  // mostly hold different cells
  const int s = max(1, (cnt + kT64 * kT64 * kT64 / 2) / (kT64 * kT64 * kT64));
  const int q = (cnt + s - 1) / s;
  // phase 1: gather, push, move; positions and amounts of the deposits go to the stash
  unsigned amax[4] = {0u, 0u, 0u, 0u};
  for (int jj = threadIdx.x; RHO && jj < q * s; jj += kThreads64) {
    const int row = jj / q, pr = (jj - row * q) * s + row;
    if (pr >= cnt) continue;
    const int64_t p = t.idx[p0 + pr];
    int64_t* st = t.stash + p0 + pr;
    const double x[3] = {a.x[p], a.y[p], a.z[p]}, qw = a.w[p] * a.qw_scale;
    bool ok = qw == 0.0 || (exponent_of(qw) >= 200 && exponent_of(qw) < 1900);
    int b[3];
    int64_t d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      ok = ok && split56<P>(x[c], a.inv_dx[c], b[c], d[c]);
      b[c] = ok ? (b[c] - T0[c] + 1) & a.mask[c] : 0;  // first node of the block in the window
      ok = ok && b[c] + NS <= kW64;
    }
    st[0] = ok ? 0 : -1;
    if (!ok) {
      push_particle_alone<P>(a, p);
      continue;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) st[(3 + c) * t.cap] = ((int64_t)b[c] << 56) | d[c];
    st[9 * t.cap] = __double_as_longlong(qw);
    amax[3] = max(amax[3], (unsigned)exponent_of(qw));
    atomicAdd(&s_blk[3 * kB64n + (b[0] * kB64 + b[1]) * kB64 + b[2]], fabsf((float)qw));
  }
  for (int jj = threadIdx.x; !RHO && jj < q * s; jj += kThreads64) {
    const int row = jj / q, pr = (jj - row * q) * s + row;
    if (pr >= cnt) continue;
    const int64_t slot = p0 + pr, p = t.idx[slot];
    const double x[3] = {a.x[p], a.y[p], a.z[p]};
    const double qw = a.w[p] * a.qw_scale;
    int g[3];
    int64_t d[3];
    bool ok = finite_bits(qw) && finite_bits(a.ux[p]) && finite_bits(a.uy[p]) && finite_bits(a.uz[p]);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      ok = ok && split56<P>(x[c], a.inv_dx[c], g[c], d[c]);
      // first node of the block, from the first staged node
      g[c] = ok ? (g[c] - T0[c]) & a.mask[c] : 0;
      ok = ok && g[c] + NS <= kG64;
    }
    if (!ok) {
      push_particle_alone<P>(a, p);
      t.stash[slot] = -1;
      continue;
    }
    double f[6];
    {
      int64_t Sx[NS], Sy[NS], Sz[NS];
      weights56<P>(d[0], Sx);
      weights56<P>(d[1], Sy);
      weights56<P>(d[2], Sz);
      Limb yz[NS][NS];
#pragma unroll
      for (int j = 0; j < NS; ++j)
#pragma unroll
        for (int k = 0; k < NS; ++k) yz[j][k] = limbs(mul56(limbs(Sy[j]), limbs(Sz[k])));
      const int4* blk = fld + (g[0] * kG64 + g[1]) * kG64 + g[2];
      // one pair of components at a time (fewer registers, a loop body a third as long)
#pragma unroll 1
      for (int r = 0; r < 3; ++r, blk += kG64n) {
        int64_t H[2] = {0, 0}, M[2] = {int64_t(1) << 27, int64_t(1) << 27};
#pragma unroll 1
        for (int i = 0; i < NS; ++i) {
          // plane sums: h, m hold the products of the high limbs and of the mixed ones (16 terms below
          // 2^58 and 2^59 each: no overflow)
          int64_t h[2] = {0, 0}, m[2] = {int64_t(1) << 27, int64_t(1) << 27};
#pragma unroll
          for (int j = 0; j < NS; ++j)
#pragma unroll
            for (int k = 0; k < NS; ++k) {
              const Limb w = yz[j][k];
              const int4 v = blk[(i * kG64 + j) * kG64 + k];
              h[0] = mad_wide(w.h, v.x, h[0]);
              h[1] = mad_wide(w.h, v.z, h[1]);
              m[0] = mad_wide(w.h, v.y, mad_wide(w.l, v.x, m[0]));
              m[1] = mad_wide(w.h, v.w, mad_wide(w.l, v.z, m[1]));
            }
          const Limb wx = limbs(Sx[i]);
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const Limb v = limbs(h[c] + (m[c] >> 28));
            H[c] = mad_wide(wx.h, v.h, H[c]);
            M[c] = mad_wide(wx.h, v.l, mad_wide(wx.l, v.h, M[c]));
          }
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) f[2 * r + c] = from_fixed(H[c] + (M[c] >> 28), (int)s_fmax[2 * r + c] - 1080);
      }
    }
    double ux, uy, uz;
    push_u(a, p, f, ux, uy, uz);
    const double ig = rsqrt(1.0 + (ux * ux + uy * uy + uz * uz) * a.inv_c2);
    const double v[3] = {ux * ig, uy * ig, uz * ig};
    int64_t* st = t.stash + slot;
    double nx[3];
    bool in = true;
    int64_t mid[3], pos[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double dd = a.dt * (v[c] - a.vg[c]);
      const double mx = wrap(x[c] + 0.5 * dd, a.L[c]);
      nx[c] = wrap(x[c] + dd, a.L[c]);
      int b;
      int64_t fr;
      in = in && split56<P>(mx, a.inv_dx[c], b, fr);
      b = (b - T0[c] + 1) & a.mask[c];  // first node of the block in the window
      in = in && b + NS <= kW64;
      mid[c] = ((int64_t)b << 56) | fr;
      in = in && split56<P>(nx[c], a.inv_dx[c], b, fr);
      b = (b - T0[c] + 1) & a.mask[c];
      in = in && b + NS <= kW64;
      pos[c] = ((int64_t)b << 56) | fr;
    }
    const double am[4] = {qw * v[0], qw * v[1], qw * v[2], qw};
#pragma unroll
    for (int c = 0; c < 4; ++c) in = in && (am[c] == 0.0 || (exponent_of(am[c]) >= 200 && exponent_of(am[c]) < 1900));
    if (!in) {  // past the window (or amounts outside 1e-247 .. 1e264): from the unchanged state, on its own
      push_particle_alone<P>(a, p);
      st[0] = -1;
      continue;
    }
    a.x[p] = nx[0];
    a.y[p] = nx[1];
    a.z[p] = nx[2];
    a.ux[p] = ux;
    a.uy[p] = uy;
    a.uz[p] = uz;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      st[c * t.cap] = mid[c];
      st[(3 + c) * t.cap] = pos[c];
    }
    const int bm = ((int)(mid[0] >> 56) * kB64 + (int)(mid[1] >> 56)) * kB64 + (int)(mid[2] >> 56);
    const int bn = ((int)(pos[0] >> 56) * kB64 + (int)(pos[1] >> 56)) * kB64 + (int)(pos[2] >> 56);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      st[(6 + c) * t.cap] = __double_as_longlong(am[c]);
      amax[c] = max(amax[c], (unsigned)exponent_of(am[c]));
      atomicAdd(&s_blk[c * kB64n + (c < 3 ? bm : bn)], fabsf((float)am[c]));
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const unsigned m = __reduce_max_sync(0xffffffffu, amax[c]);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_amax[c], m);
  }
  __syncthreads();
  // the units of the four sums, 2^(ref - 1080): every node's sum < 2^63 units (the bound has 1 % to spare); where the FP32 bound is
  // out of that type's range, from the count of particles
  node_bounds<P, RHO ? 3 : 0>(s_blk, reinterpret_cast<float*>(smraw64), s_bound);
  int ref[4];
  {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float b = __uint_as_float(s_bound[c]) * 1.01f;
      ref[c] = (b > 1e-30f && b < 1e30f) ? (int)(__float_as_uint(b) >> 23) - 127 + 1023 - 5
                                         : (int)s_amax[c] + 32 - __clz(cnt) - 5;
      ref[c] = max(ref[c], (int)s_amax[c] - kRowShift<P> - 3);  // (see deposit56)
    }
  }
  // the staged fields are dead: clear the window in their place
  uint32_t* win = reinterpret_cast<uint32_t*>(smraw64);
  for (int e = threadIdx.x; e < 2 * kW64n; e += kThreads64) reinterpret_cast<uint4*>(win)[e] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  // phase 2: deposits (same thread, same particles)
  for (int jj = threadIdx.x; jj < q * s; jj += kThreads64) {
    const int row = jj / q, pr = (jj - row * q) * s + row;
    if (pr >= cnt) continue;
    const int64_t* st = t.stash + p0 + pr;
    int64_t pos[3], am[3];
    int l[3];
    // amounts of window components c0 .. c0 + nc - 1
    int lz;
    const auto amounts = [&](int c0, int nc) {
      double v[3];
      lz = 0;
      for (int c = 0; c < nc; ++c) {
        v[c] = __longlong_as_double(st[(6 + c0 + c) * t.cap]);
        l[c] = max(0, exponent_of(v[c]) - ref[c0 + c]);
        lz = max(lz, l[c] - kRowShift<P>);
      }
      for (int c = 0; c < nc; ++c) {
        l[c] = max(l[c] - lz, 0);
        am[c] = to_fixed58(v[c], ref[c0 + c] + l[c] + lz);
      }
    };
    pos[0] = st[0];
    if (pos[0] < 0) continue;
    if constexpr (!RHO) {
      pos[1] = st[t.cap];
      pos[2] = st[2 * t.cap];
      amounts(0, 3);
      deposit56<P, 3>(win, 0, pos, am, l, lz);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) pos[c] = st[(3 + c) * t.cap];
    amounts(3, 1);
    deposit56<P, 1>(win, 3, pos, am, l, lz);
  }
  __syncthreads();
  double* dst[4] = {a.J[0], a.J[1], a.J[2], a.rho};
  for (int e = threadIdx.x; e < kW64n; e += kThreads64) {
    const int k = e % kW64, r = e / kW64, j = r % kW64, i = r / kW64;
    const int o = (((T0[0] - 2 + i) & a.mask[0]) * Ny + ((T0[1] - 2 + j) & a.mask[1])) * Nz + ((T0[2] - 2 + k) & a.mask[2]);
#pragma unroll
    for (int c = RHO ? 3 : 0; c < 4; ++c) {
      const int64_t v = (int64_t)(((uint64_t)win[(4 + c) * kW64n + e] << 32) | win[c * kW64n + e]);
      if (v != 0) atomicAdd(dst[c] + o, from_fixed(v, ref[c] - 1080));
    }
  }
}

// particle numbers grouped by tile: tile of every particle and the tiles' counts
struct Tile64List {
  PushArgs a;
  int nt[3];
  int n_tiles;
  int chunk;        // particles per chunk at most
  int32_t* tid;
  int32_t* count;   // [n_tiles], cleared
  int32_t* off;     // [n_tiles + 1]
  int32_t* cursor;  // [n_tiles], cleared
  int32_t* cstart;  // [n_tiles + 1]
  int32_t* ctile;
  int32_t* idx;
};

__global__ void tile64_count_kernel(Tile64List l) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= l.a.n) return;
  const double* x[3] = {l.a.x, l.a.y, l.a.z};
  int c[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    int64_t fr;
    c[d] = 0;
    if (!split56<1>(x[d][p], l.a.inv_dx[d], c[d], fr)) c[d] = 0;  // such a particle is pushed on its own
    c[d] = (c[d] & l.a.mask[d]) / kT64;
  }
  const int t = (c[0] * l.nt[1] + c[1]) * l.nt[2] + c[2];
  l.tid[p] = t;
  const unsigned peers = __match_any_sync(__activemask(), t);
  if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(l.count + t, __popc(peers));
}

// exclusive scans of the counts and of the tiles' chunk counts, and the tile of every chunk (one CTA)
__global__ void __launch_bounds__(1024) tile64_scan_kernel(Tile64List l) {
  __shared__ int2 part[1024];
  const int per = (l.n_tiles + 1023) / 1024;
  const int b = min(l.n_tiles, (int)threadIdx.x * per), e = min(l.n_tiles, b + per);
  int2 s = make_int2(0, 0);
  for (int i = b; i < e; ++i) {
    const int n = l.count[i];
    s.x += n;
    s.y += (n + l.chunk - 1) / l.chunk;
  }
  part[threadIdx.x] = s;
  __syncthreads();
  for (int d = 1; d < 1024; d <<= 1) {
    const int2 v = threadIdx.x >= d ? part[threadIdx.x - d] : make_int2(0, 0);
    __syncthreads();
    part[threadIdx.x].x += v.x;
    part[threadIdx.x].y += v.y;
    __syncthreads();
  }
  int2 run = threadIdx.x > 0 ? part[threadIdx.x - 1] : make_int2(0, 0);
  for (int i = b; i < e; ++i) {
    const int n = l.count[i];
    l.off[i] = run.x;
    l.cstart[i] = run.y;
    l.cursor[i] = run.x;
    const int nch = (n + l.chunk - 1) / l.chunk;
    for (int k = 0; k < nch; ++k) l.ctile[run.y + k] = i;
    run.x += n;
    run.y += nch;
  }
  if (threadIdx.x == 1023) {
    l.off[l.n_tiles] = part[1023].x;
    l.cstart[l.n_tiles] = part[1023].y;
  }
}

__global__ void tile64_list_kernel(Tile64List l) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= l.a.n) return;
  const int t = l.tid[p];
  const unsigned peers = __match_any_sync(__activemask(), t);
  const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(l.cursor + t, __popc(peers));
  base = __shfl_sync(peers, base, leader);
  l.idx[base + __popc(peers & ((1u << lane) - 1u))] = (int32_t)p;
}

PushArgs make_args(pic_ctx* ctx, const pic_species* sp) {
  PushArgs a;
  a.x = sp->x;
  a.y = sp->y;
  a.z = sp->z;
  a.ux = sp->ux;
  a.uy = sp->uy;
  a.uz = sp->uz;
  a.w = sp->w;
  a.n = sp->n;
  for (int d = 0; d < 3; ++d) {
    a.inv_dx[d] = 1.0 / ctx->dx[d];
    a.L[d] = (double)ctx->N[d] * ctx->dx[d];
    a.mask[d] = (int)ctx->N[d] - 1;
    a.vg[d] = ctx->variant == PIC_PSATD_STANDARD ? 0.0 : ctx->vg[d];
  }
  a.Ny = ctx->N[1];
  a.Nz = ctx->N[2];
  a.qm_half_dt = sp->q * ctx->dt / (2.0 * sp->m);
  a.dt = ctx->dt;
  a.inv_c2 = 1.0 / (ctx->c * ctx->c);
  a.vay = ctx->pusher == PIC_PUSHER_VAY ? 1 : 0;
  a.qw_scale = sp->q / (ctx->dx[0] * ctx->dx[1] * ctx->dx[2]);
  return a;
}

// The tiled push covers orders 2 and 3 (at order 1 the node sums are a fifth of the FP64 operations and
// the lists cost what they save) on the nodal grid, for species with at least 4 particles per tile on
// average: below that most tiles hold too few to be worth staging.
int tiles64(const pic_ctx* ctx) {
  return (int)((ctx->N[0] / kT64) * (ctx->N[1] / kT64) * (ctx->N[2] / kT64));
}
bool use_tiled64(const pic_ctx* ctx, int64_t n) {
  return ctx->shape_order >= 2 && ctx->cycle != PIC_CYCLE_STAGGERED && n >= 4 * (int64_t)tiles64(ctx);
}

// scratch for n particles, kept by the context; false (and no error) when there is none: not enough
// memory, or the stream is being captured, where nothing may be allocated
bool tiled64_scratch(pic_ctx* ctx, int64_t n) {
  if (ctx->t64_cap >= n) return true;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(ctx->stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return false;
  // It at least doubles as it grows, and the outgrown arrays live until the context is destroyed: a
  // captured graph of an earlier call may still use them.
  if (ctx->t64_nold + 2 > kT64Old) return false;
  n = std::max(n, 2 * ctx->t64_cap);
  const size_t nt = (size_t)tiles64(ctx), words = 2 * (size_t)n + 5 * nt + 2 + (size_t)n / kChunk64Min + 1;
  int32_t* w = nullptr;
  int64_t* st = nullptr;
  if (cudaMalloc(&w, words * sizeof(int32_t)) != cudaSuccess ||
      cudaMalloc(&st, 10 * (size_t)n * sizeof(int64_t)) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(w);
    return false;
  }
  if (ctx->t64_cap > 0) {
    ctx->t64_old[ctx->t64_nold++] = ctx->t64_int;
    ctx->t64_old[ctx->t64_nold++] = ctx->t64_stash;
  }
  ctx->t64_int = w;
  ctx->t64_stash = st;
  ctx->t64_cap = n;
  return true;
}

template <int P, bool RHO>
pic_status launch_push64_tiled(pic_ctx* ctx, const PushArgs& a) {
  const int nt = tiles64(ctx);
  const int64_t cap = ctx->t64_cap;
  Tile64List l;
  l.a = a;
  Tile64Args t;
  for (int d = 0; d < 3; ++d) l.nt[d] = t.nt[d] = (int)ctx->N[d] / kT64;
  l.n_tiles = t.n_tiles = nt;
  int32_t* w = ctx->t64_int;
  l.count = w;
  l.cursor = l.count + nt;
  l.off = l.cursor + nt;
  l.cstart = l.off + nt + 1;
  l.tid = l.cstart + nt + 1;
  l.idx = l.tid + cap;
  l.ctile = l.idx + cap;  // [nt + cap / kChunk64Min + 1]
  // about two chunks per resident CTA (two per SM) of a small species; 131072 cubic particles on 32^3, in 64
  // tiles: 64 chunks of 2048 kept 64 of 304 CTAs busy (the gradient over 8 steps there 15.16 -> 13.62 ms)
  l.chunk = (int)std::min<int64_t>(kChunk64, std::max<int64_t>(kChunk64Min, a.n / (4 * std::max(1, ctx->nsm))));
  t.idx = l.idx;
  t.off = l.off;
  t.cstart = l.cstart;
  t.ctile = l.ctile;
  t.stash = ctx->t64_stash;
  t.cap = cap;
  const unsigned nb = (unsigned)((a.n + 255) / 256);
  PIC_CUDA_TRY(ctx, cudaMemsetAsync(l.count, 0, nt * sizeof(int32_t), ctx->stream));
  tile64_count_kernel<<<nb, 256, 0, ctx->stream>>>(l);
  PIC_LAUNCH_CHECK(ctx);
  tile64_scan_kernel<<<1, 1024, 0, ctx->stream>>>(l);
  PIC_LAUNCH_CHECK(ctx);
  tile64_list_kernel<<<nb, 256, 0, ctx->stream>>>(l);
  PIC_LAUNCH_CHECK(ctx);
  PIC_CUDA_TRY(ctx, cudaFuncSetAttribute(push64_tile_kernel<P, RHO>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem64));
  // sum over tiles of ceil(count / chunk) <= n_tiles + n / chunk: surplus CTAs return at once
  push64_tile_kernel<P, RHO><<<(unsigned)(nt + a.n / l.chunk + 1), kThreads64, kSmem64, ctx->stream>>>(a, t);
  PIC_LAUNCH_CHECK(ctx);
  return PIC_OK;
}

pic_status launch_push(pic_ctx* ctx, const PushArgs& a) {
  if (a.n == 0) return PIC_OK;
  if (a.gather && use_tiled64(ctx, a.n) && tiled64_scratch(ctx, a.n))
    return ctx->shape_order == 2 ? launch_push64_tiled<2, false>(ctx, a) : launch_push64_tiled<3, false>(ctx, a);
  if (!a.gather && use_tiled64(ctx, a.n) && a.n >= kMinRho64 && tiled64_scratch(ctx, a.n))
    return ctx->shape_order == 2 ? launch_push64_tiled<2, true>(ctx, a) : launch_push64_tiled<3, true>(ctx, a);
  const int bs = 256;
  const unsigned nb = (unsigned)((a.n + bs - 1) / bs);
  if (a.gather && ctx->cycle == PIC_CYCLE_STAGGERED) {
    switch (ctx->shape_order) {
      case 1: push_stag_kernel<1><<<nb, bs, 0, ctx->stream>>>(a); break;
      case 2: push_stag_kernel<2><<<nb, bs, 0, ctx->stream>>>(a); break;
      default: push_stag_kernel<3><<<nb, bs, 0, ctx->stream>>>(a); break;
    }
    PIC_LAUNCH_CHECK(ctx);
    return PIC_OK;
  }
  switch (ctx->shape_order) {
    case 1: push_kernel<1><<<nb, bs, 0, ctx->stream>>>(a); break;
    case 2: push_kernel<2><<<nb, bs, 0, ctx->stream>>>(a); break;
    default: push_kernel<3><<<nb, bs, 0, ctx->stream>>>(a); break;
  }
  PIC_LAUNCH_CHECK(ctx);
  return PIC_OK;
}

// ---------------------------------------------------------------------------
// tile binning
// ---------------------------------------------------------------------------
struct BinArgs {
  const double *x, *y, *z;
  int64_t n;
  double inv_dx[3];
  int mask[3];
  int tshift[3];  // log2 of the tile edge
  int64_t nty, ntz;
  int32_t* tid;
  unsigned long long* counts;
};

__global__ void tile_id_kernel(BinArgs a) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= a.n) return;
  const int cx = (int)floor(__dmul_rn(a.x[p], a.inv_dx[0])) & a.mask[0];
  const int cy = (int)floor(__dmul_rn(a.y[p], a.inv_dx[1])) & a.mask[1];
  const int cz = (int)floor(__dmul_rn(a.z[p], a.inv_dx[2])) & a.mask[2];
  const int t = (int)(((cx >> a.tshift[0]) * a.nty + (cy >> a.tshift[1])) * a.ntz + (cz >> a.tshift[2]));
  a.tid[p] = t;
  // warp-aggregated histogram
  const unsigned active = __activemask();
  const unsigned peers = __match_any_sync(active, t);
  const int leader = __ffs(peers) - 1;
  if ((int)(threadIdx.x & 31) == leader) atomicAdd(a.counts + t, (unsigned long long)__popc(peers));
}

// Exclusive scan of n counts into off[0..n] by one CTA (n up to a few million).
__global__ void __launch_bounds__(1024) scan_kernel(const unsigned long long* cnt, int64_t* off, int64_t n) {
  __shared__ unsigned long long part[1024];
  const int T = blockDim.x;
  const int64_t chunk = (n + T - 1) / T;
  const int64_t b = threadIdx.x * chunk, e = min(n, b + chunk);
  unsigned long long s = 0;
  for (int64_t i = b; i < e; ++i) s += cnt[i];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int d = 1; d < T; d <<= 1) {
    unsigned long long v = threadIdx.x >= d ? part[threadIdx.x - d] : 0ull;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  unsigned long long run = threadIdx.x > 0 ? part[threadIdx.x - 1] : 0ull;
  for (int64_t i = b; i < e; ++i) {
    off[i] = (int64_t)run;
    run += cnt[i];
  }
  if (threadIdx.x == T - 1) off[n] = (int64_t)part[T - 1];
}

struct ScatterArgs {
  const double* src[8];  // x y z ux uy uz w id(as double bits)
  double* dst[8];
  int nfield;
  int64_t n;
  const int32_t* tid;
  const int64_t* off;
  unsigned long long* cursor;
};

__global__ void scatter_kernel(ScatterArgs a) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= a.n) return;
  const int t = a.tid[p];
  const unsigned active = __activemask();
  const unsigned peers = __match_any_sync(active, t);
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(peers) - 1;
  const int rank = __popc(peers & ((1u << lane) - 1u));
  unsigned long long base = 0;
  if (lane == leader) base = atomicAdd(a.cursor + t, (unsigned long long)__popc(peers));
  base = __shfl_sync(peers, base, leader);
  const int64_t q = a.off[t] + (int64_t)base + rank;
  for (int f = 0; f < a.nfield; ++f) a.dst[f][q] = a.src[f][p];
}

pic_status ensure_bin_capacity(pic_ctx* ctx, int64_t n) {
  if (ctx->bin_counts == nullptr) {
    PIC_CUDA_TRY(ctx, cudaMalloc(&ctx->bin_counts, (ctx->n_tiles + 1) * sizeof(int64_t)));
    PIC_CUDA_TRY(ctx, cudaMalloc(&ctx->bin_cursor, ctx->n_tiles * sizeof(int64_t)));
  }
  if (n <= ctx->bin_cap) return PIC_OK;
  cudaFree(ctx->bin_tid);
  cudaFree(ctx->bin_tmp);
  ctx->bin_tid = nullptr;
  ctx->bin_tmp = nullptr;
  ctx->bin_cap = 0;
  if (cudaMalloc(&ctx->bin_tid, n * sizeof(int32_t)) != cudaSuccess ||
      cudaMalloc(&ctx->bin_tmp, 8 * n * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    return pic_set_error(ctx, PIC_ERR_NOMEM, "binning scratch for %lld particles", (long long)n);
  }
  ctx->bin_cap = n;
  return PIC_OK;
}

int ilog2(int v) {
  int r = 0;
  while ((1 << r) < v) ++r;
  return r;
}

}  // namespace

int particles_push_launches(const pic_ctx* ctx, int64_t n) { return n == 0 ? 0 : (use_tiled64(ctx, n) ? 4 : 1); }

pic_status particles_bin_capacity(pic_ctx* ctx, int64_t n) { return ensure_bin_capacity(ctx, n); }

pic_status particles_push(pic_ctx* ctx, const double* const En[3], const double* const Bn[3],
                          const pic_species* sp, double* const J[3], double* rho) {
  PushArgs a = make_args(ctx, sp);
  for (int c = 0; c < 3; ++c) {
    a.F[c] = En[c];
    a.F[3 + c] = Bn[c];
    a.J[c] = J[c];
  }
  a.rho = rho;
  a.gather = 1;
  return launch_push(ctx, a);
}

pic_status particles_deposit_rho(pic_ctx* ctx, const pic_species* sp, double* rho) {
  PushArgs a = make_args(ctx, sp);
  for (int c = 0; c < 6; ++c) a.F[c] = nullptr;
  for (int c = 0; c < 3; ++c) a.J[c] = nullptr;
  a.rho = rho;
  a.gather = 0;
  return launch_push(ctx, a);
}

pic_status particles_bin(pic_ctx* ctx, const pic_species* sp, int64_t* offsets_out) {
  const int64_t n = sp->n;
  pic_status st = ensure_bin_capacity(ctx, n > 0 ? n : 1);
  if (st != PIC_OK) return st;
  unsigned long long* cnt = reinterpret_cast<unsigned long long*>(ctx->bin_cursor);
  PIC_CUDA_TRY(ctx, cudaMemsetAsync(cnt, 0, ctx->n_tiles * sizeof(int64_t), ctx->stream));
  BinArgs b;
  b.x = sp->x;
  b.y = sp->y;
  b.z = sp->z;
  b.n = n;
  for (int d = 0; d < 3; ++d) {
    b.inv_dx[d] = 1.0 / ctx->dx[d];
    b.mask[d] = (int)ctx->N[d] - 1;
    b.tshift[d] = ilog2(ctx->tile[d]);
  }
  b.nty = ctx->N[1] / ctx->tile[1];
  b.ntz = ctx->N[2] / ctx->tile[2];
  b.tid = ctx->bin_tid;
  b.counts = cnt;
  const int bs = 256;
  const unsigned nb = (unsigned)((n + bs - 1) / bs);
  if (n > 0) {
    tile_id_kernel<<<nb, bs, 0, ctx->stream>>>(b);
    PIC_LAUNCH_CHECK(ctx);
  }
  scan_kernel<<<1, 1024, 0, ctx->stream>>>(cnt, ctx->bin_counts, ctx->n_tiles);
  PIC_LAUNCH_CHECK(ctx);
  if (offsets_out)
    PIC_CUDA_TRY(ctx, cudaMemcpyAsync(offsets_out, ctx->bin_counts, (ctx->n_tiles + 1) * sizeof(int64_t),
                                      cudaMemcpyDeviceToDevice, ctx->stream));
  if (n == 0) return PIC_OK;
  PIC_CUDA_TRY(ctx, cudaMemsetAsync(cnt, 0, ctx->n_tiles * sizeof(int64_t), ctx->stream));
  ScatterArgs s;
  double* fields[8] = {sp->x, sp->y, sp->z, sp->ux, sp->uy, sp->uz, sp->w, reinterpret_cast<double*>(sp->id)};
  s.nfield = sp->id ? 8 : 7;
  for (int f = 0; f < s.nfield; ++f) {
    s.src[f] = fields[f];
    s.dst[f] = ctx->bin_tmp + (int64_t)f * ctx->bin_cap;
  }
  s.n = n;
  s.tid = ctx->bin_tid;
  s.off = ctx->bin_counts;
  s.cursor = cnt;
  scatter_kernel<<<nb, bs, 0, ctx->stream>>>(s);
  PIC_LAUNCH_CHECK(ctx);
  for (int f = 0; f < s.nfield; ++f)
    PIC_CUDA_TRY(ctx, cudaMemcpyAsync(fields[f], s.dst[f], n * sizeof(double), cudaMemcpyDeviceToDevice,
                                      ctx->stream));
  return PIC_OK;
}
