// Reverse mode of the FP64 hybrid PIC step (pic_adjoint_step).
//
// The step is a composition of maps; its adjoint applies the transpose of each
// in reverse order: the PSATD update (per-mode conjugate transpose of the
// coefficient matrix, psatd.cu), the J centering (transpose = multiplication by
// zeta on the nodal spectrum), the deposits (transpose = gather of the adjoint
// densities, plus the B-spline derivative for positions), the move and v = u /
// gamma, the Boris push (reverse chain rule through its intermediates), the
// gather (transpose = deposit of the force adjoints, plus the shape derivative)
// and the E, B centering (transpose = zeta on the adjoint spectra).  Every
// forward quantity a transpose needs is recomputed from the state at t^n.
#include "pic_internal.cuh"

#include <algorithm>

namespace {

constexpr int kAdjThreads = 64;

struct AdjArgs {
  const double *x, *y, *z, *ux, *uy, *uz, *w;
  double *xb, *yb, *zb, *uxb, *uyb, *uzb;  // in: adjoints of x^{n+1}, u^{n+1/2}; out: of x^n, u^{n-1/2}
  int64_t n;
  const double* F[6];    // nodal E, B at t^n
  const double* Jb[3];   // nodal adjoint of J^{n+1/2}
  const double* Rb;      // nodal adjoint of rho^{n+1}
  double* Fb[6];         // nodal adjoints of the gathered E, B (atomic add)
  double inv_dx[3];
  double L[3];
  int mask[3];
  int64_t Ny, Nz;
  double k;              // q dt / (2 m)
  double dt;
  double inv_c2;
  double vg[3];
  double qw_scale;       // q / dV
};

// B-spline weights and their derivative along the axis (per cell), same cell rule as the forward.
template <int P>
__device__ __forceinline__ void shape_d(double x, double inv, int& lo, double* S, double* D) {
  const double t = __dmul_rn(x, inv);
  int b;
  const double d = t - floor_cell(P == 2 ? __dadd_rn(t, 0.5) : t, b);
  if (P == 1) {
    lo = b;
    S[0] = 1.0 - d;
    S[1] = d;
    D[0] = -1.0;
    D[1] = 1.0;
  } else if (P == 2) {
    lo = b - 1;
    const double a = 0.5 - d, c = 0.5 + d;
    S[0] = 0.5 * a * a;
    S[1] = 0.75 - d * d;
    S[2] = 0.5 * c * c;
    D[0] = -a;
    D[1] = -2.0 * d;
    D[2] = c;
  } else {
    // the inner weights as 2/3 + d^2 (d/2 - 1) and its mirror image: 17 operations with the derivatives
    lo = b - 1;
    const double e = 1.0 - d, d2 = d * d, e2 = e * e;
    S[0] = e2 * (e * (1.0 / 6.0));
    S[1] = fma(d2, fma(0.5, d, -1.0), 2.0 / 3.0);
    S[2] = fma(e2, fma(0.5, e, -1.0), 2.0 / 3.0);
    S[3] = d2 * (d * (1.0 / 6.0));
    D[0] = -0.5 * e2;
    D[1] = d * fma(1.5, d, -2.0);
    D[2] = e * fma(-1.5, e, 2.0);
    D[3] = 0.5 * d2;
  }
}

// x >= L: x - L; x < 0: x + L, the comparisons on the bit patterns (off the FP64 pipe; L > 0)
__device__ __forceinline__ double wrapd(double x, double L) {
  const long long b = __double_as_longlong(x);
  if (b >= __double_as_longlong(L)) return x - L;
  if (b < 0 && (b << 1) != 0) return x + L;
  return x;
}

// Value and gradient (per cell) of a nodal array at a position, from the first nodes and the weights S and
// their derivatives D of the three axes, one axis after the other: a z row gives its sum with Sz and with
// Dz, a plane three sums, the block four.  The FP64 pipe (1.7 operations per clock and SM) bounds the
// kernel: 2 P' + 3 / P' + 4 / P'^2 operations per node (P' = P + 1) and array, where four products of three
// weights and four multiply-adds per node took 6 to 7; cubic 192 instead of about 330 per array.  Linear:
// differences along the axis, which are the derivative and give the value by one multiply-add each, 22
// operations instead of 36.  f(j, k, s, o): the array at node (j, k) of the plane of weight s, o its index.
// The planes of orders 2 and 3 are a rolled loop, their weights in shared memory (wx: per thread Sx, Dx).
template <int P, bool VAL, class Fn>
__device__ __forceinline__ void node_grad(const AdjArgs& a, const int* lo, const double (*S)[P + 1],
                                          const double (*D)[P + 1], const double* wx, double& val, double* grad,
                                          Fn&& f) {
  constexpr int NS = P + 1;
  double p0 = 0.0, py0 = 0.0, pz0 = 0.0;  // linear: the first plane's sums
  if (VAL) val = 0.0;
  grad[0] = grad[1] = grad[2] = 0.0;
#pragma unroll (P == 1 ? 2 : 1)
  for (int i = 0; i < NS; ++i) {
    const double Sx = P == 1 ? S[0][i] : wx[i * kAdjThreads], Dx = P == 1 ? 0.0 : wx[(NS + i) * kAdjThreads];
    const int64_t ox = (int64_t)((lo[0] + i) & a.mask[0]) * a.Ny;
    double p = 0.0, py = 0.0, pz = 0.0;  // the plane's sums: S, d/dy, d/dz
    double r0 = 0.0, rz0 = 0.0;          // linear: the first row's
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      const int64_t oy = (ox + ((lo[1] + j) & a.mask[1])) * a.Nz;
      double r = 0.0, rz = 0.0;
      if constexpr (P == 1) {
        const double f0 = f(j, 0, Sx, oy + (lo[2] & a.mask[2])), f1 = f(j, 1, Sx, oy + ((lo[2] + 1) & a.mask[2]));
        rz = f1 - f0;
        r = fma(S[2][1], rz, f0);
        if (j == 0) {
          r0 = r;
          rz0 = rz;
        } else {
          py = r - r0;
          p = fma(S[1][1], py, r0);
          pz = fma(S[1][1], rz - rz0, rz0);
        }
      } else {
#pragma unroll
        for (int k = 0; k < NS; ++k) {
          const double v = f(j, k, Sx, oy + ((lo[2] + k) & a.mask[2]));
          r = k == 0 ? S[2][0] * v : fma(S[2][k], v, r);
          rz = k == 0 ? D[2][0] * v : fma(D[2][k], v, rz);
        }
        p = j == 0 ? S[1][0] * r : fma(S[1][j], r, p);
        py = j == 0 ? D[1][0] * r : fma(D[1][j], r, py);
        pz = j == 0 ? S[1][0] * rz : fma(S[1][j], rz, pz);
      }
    }
    if constexpr (P == 1) {
      if (i == 0) {
        p0 = p;
        py0 = py;
        pz0 = pz;
      } else {
        grad[0] = p - p0;
        if (VAL) val = fma(S[0][1], grad[0], p0);
        grad[1] = fma(S[0][1], py - py0, py0);
        grad[2] = fma(S[0][1], pz - pz0, pz0);
      }
    } else {
      if (VAL) val = fma(Sx, p, val);
      grad[0] = fma(Dx, p, grad[0]);
      grad[1] = fma(Sx, py, grad[1]);
      grad[2] = fma(Sx, pz, grad[2]);
    }
  }
}
template <int P, bool VAL>
__device__ __forceinline__ void gather_grad(const AdjArgs& a, const double* __restrict__ F, const int* lo,
                                            const double (*S)[P + 1], const double (*D)[P + 1], const double* wx,
                                            double& val, double* grad) {
  node_grad<P, VAL>(a, lo, S, D, wx, val, grad, [&](int, int, double, int64_t o) { return __ldg(F + o); });
}

// value only
template <int P>
__device__ __forceinline__ double gather_value(const AdjArgs& a, const double* __restrict__ F, const int* lo,
                                               const double (*S)[P + 1], const double* wx) {
  constexpr int NS = P + 1;
  double val = 0.0;
#pragma unroll 1
  for (int i = 0; i < NS; ++i) {
    const int64_t ox = (int64_t)((lo[0] + i) & a.mask[0]) * a.Ny;
    double p = 0.0;
#pragma unroll
    for (int j = 0; j < NS; ++j) {
      const int64_t oy = (ox + ((lo[1] + j) & a.mask[1])) * a.Nz;
      double r = 0.0;
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        const double v = __ldg(F + oy + ((lo[2] + k) & a.mask[2]));
        r = k == 0 ? S[2][0] * v : fma(S[2][k], v, r);
      }
      p = j == 0 ? S[1][0] * r : fma(S[1][j], r, p);
    }
    val = fma(wx[i * kAdjThreads], p, val);
  }
  return val;
}

// first nodes, weights and derivatives at a position; those of x also to the thread's shared-memory column
template <int P>
__device__ __forceinline__ void shapes_d(const AdjArgs& a, const double* x, int* lo, double (*S)[P + 1],
                                         double (*D)[P + 1], double* wx) {
#pragma unroll
  for (int c = 0; c < 3; ++c) shape_d<P>(x[c], a.inv_dx[c], lo[c], S[c], D[c]);
  if (P > 1) {
#pragma unroll
    for (int i = 0; i <= P; ++i) {
      wx[i * kAdjThreads] = S[0][i];
      wx[(P + 1 + i) * kAdjThreads] = D[0][i];
    }
  }
}

__device__ __forceinline__ void cross3(const double* a, const double* b, double* o) {
  o[0] = a[1] * b[2] - a[2] * b[1];
  o[1] = a[2] * b[0] - a[0] * b[2];
  o[2] = a[0] * b[1] - a[1] * b[0];
}

// o = base + a x b
__device__ __forceinline__ void cross3_add(const double* base, const double* a, const double* b, double* o) {
  o[0] = fma(a[1], b[2], fma(-a[2], b[1], base[0]));
  o[1] = fma(a[2], b[0], fma(-a[0], b[2], base[1]));
  o[2] = fma(a[0], b[1], fma(-a[1], b[0], base[2]));
}

// One thread per particle; 64-thread CTAs, so that the FP64-bound work of a small species spreads evenly
// over the SMs.  Divisions by gamma, gamma^{n+1/2} and 1 + t^2 are one rsqrt or reciprocal each and
// products (an FP64 division costs about ten operations; there were 25).  The FP64 pipe bounds it (84-86%
// of its peak with 8 to 12 warps per SM; more warps changed nothing), so a pass is as long as its operations:
// cubic 2870 -> 2706, linear 686 -> 522 per particle, one reverse step of 131072 cubic ones on 32^3
// 0.83 -> 0.67 ms, of 1.05 million linear ones on 64^3 1.39 -> 1.05 ms.
template <int P>
__global__ void __launch_bounds__(kAdjThreads) adjoint_push_kernel(AdjArgs a) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= a.n) return;
  constexpr int NS = P + 1;
  const double x[3] = {a.x[p], a.y[p], a.z[p]};
  const double u[3] = {a.ux[p], a.uy[p], a.uz[p]};
  const double qw = a.w[p] * a.qw_scale;
  int lo[3];
  double S[3][NS], D[3][NS];
  // per thread: Sx, Dx of the current position; Sx, Dx, Sy, ... Dz of x^n, which is needed twice
  __shared__ double s_wx[P == 1 ? 1 : 8 * NS * kAdjThreads];
  double* const wx = s_wx + (P == 1 ? 0 : threadIdx.x);
  double* const w0 = wx + 2 * NS * kAdjThreads;
  int lo0[3];
  double d0[3];
  // forward recompute: gather (with gradients) and Boris
  double F[6], dF[P == 1 ? 6 : 1][3];
  shapes_d<P>(a, x, lo, S, D, wx);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    lo0[c] = lo[c];
    if constexpr (P == 1) {
      d0[c] = S[c][1];
    } else {
#pragma unroll
      for (int i = 0; i < NS; ++i) {
        w0[(2 * c * NS + i) * kAdjThreads] = S[c][i];
        w0[((2 * c + 1) * NS + i) * kAdjThreads] = D[c][i];
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    if constexpr (P == 1) gather_grad<P, true>(a, a.F[c], lo, S, D, wx, F[c], dF[c]);
    else F[c] = gather_value<P>(a, a.F[c], lo, S, wx);
  }
  const double k = a.k;
  double um[3], t[3], s[3], up[3], un[3];
  for (int c = 0; c < 3; ++c) um[c] = u[c] + k * F[c];
  const double igm = rsqrt(1.0 + (um[0] * um[0] + um[1] * um[1] + um[2] * um[2]) * a.inv_c2);
  for (int c = 0; c < 3; ++c) t[c] = k * F[3 + c] * igm;
  const double s2 = 2.0 / (1.0 + t[0] * t[0] + t[1] * t[1] + t[2] * t[2]);
  for (int c = 0; c < 3; ++c) s[c] = s2 * t[c];
  double tmp[3];
  cross3_add(um, um, t, up);
  for (int c = 0; c < 3; ++c) tmp[c] = um[c] + k * F[c];
  cross3_add(tmp, up, s, un);
  const double ig = rsqrt(1.0 + (un[0] * un[0] + un[1] * un[1] + un[2] * un[2]) * a.inv_c2);
  double v[3], mid[3], nw[3];
  for (int c = 0; c < 3; ++c) {
    v[c] = un[c] * ig;
    const double dd = a.dt * (v[c] - a.vg[c]);
    mid[c] = wrapd(x[c] + 0.5 * dd, a.L[c]);
    nw[c] = wrapd(x[c] + dd, a.L[c]);
  }
  // deposits, reversed: gather the adjoint densities (and gradients) at x^{n+1/2}, x^{n+1}
  double Jv[3], dJ[3][3], dR[3], none;
  shapes_d<P>(a, mid, lo, S, D, wx);
#pragma unroll
  for (int c = 0; c < 3; ++c) gather_grad<P, true>(a, a.Jb[c], lo, S, D, wx, Jv[c], dJ[c]);
  shapes_d<P>(a, nw, lo, S, D, wx);
  gather_grad<P, false>(a, a.Rb, lo, S, D, wx, none, dR);
  double xnb[3], xmb[3], vb[3], xb[3];
  const double xin[3] = {a.xb[p], a.yb[p], a.zb[p]};
  for (int c = 0; c < 3; ++c) {
    const double qi = qw * a.inv_dx[c];
    xnb[c] = xin[c] + qi * dR[c];
    xmb[c] = qi * (v[0] * dJ[0][c] + v[1] * dJ[1][c] + v[2] * dJ[2][c]);
    vb[c] = qw * Jv[c] + 0.5 * a.dt * xmb[c] + a.dt * xnb[c];
    xb[c] = xnb[c] + xmb[c];
  }
  // v = u / gamma
  const double udv = (un[0] * vb[0] + un[1] * vb[1] + un[2] * vb[2]) * a.inv_c2 * (ig * ig * ig);
  const double unb[3] = {a.uxb[p] + vb[0] * ig - un[0] * udv, a.uyb[p] + vb[1] * ig - un[1] * udv,
                         a.uzb[p] + vb[2] * ig - un[2] * udv};
  // Boris, reversed
  double Eb[3], Bb[3], umb[3], upb[3], sb[3], tb[3];
  for (int c = 0; c < 3; ++c) Eb[c] = k * unb[c];
  cross3(s, unb, upb);        // upl = um + up x s
  cross3(unb, up, sb);
  for (int c = 0; c < 3; ++c) tmp[c] = unb[c] + upb[c];
  cross3_add(tmp, t, upb, umb);  // up = um + um x t
  cross3(upb, um, tb);
  const double sdt = sb[0] * t[0] + sb[1] * t[1] + sb[2] * t[2];
  for (int c = 0; c < 3; ++c) tb[c] += s2 * sb[c] - s2 * s2 * sdt * t[c];
  for (int c = 0; c < 3; ++c) Bb[c] = k * igm * tb[c];
  const double gmb = -(t[0] * tb[0] + t[1] * tb[1] + t[2] * tb[2]) * igm;
  const double gmc = gmb * a.inv_c2 * igm;
  for (int c = 0; c < 3; ++c) umb[c] += gmc * um[c];
  for (int c = 0; c < 3; ++c) Eb[c] += k * umb[c];
  // gather, reversed: deposit the force adjoints at x^n, node (i, j, k) receiving (Sx_i fb)(Sy_j Sz_k), one
  // product per node and array; and the shape derivative of sum_c fb_c F_c for the position.  The adjoints
  // fb are known only here, so orders 2 and 3 read F again and form that sum at the nodes (cubic: 6 84 + 384
  // + 188 operations instead of 6 192, and no 18 gradients kept); the linear gradients are the cheaper ones
  const double fb[6] = {Eb[0], Eb[1], Eb[2], Bb[0], Bb[1], Bb[2]};
  double yz[NS][NS], fx[6], grad[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    lo[c] = lo0[c];
    if constexpr (P == 1) {
      S[c][0] = 1.0 - d0[c];
      S[c][1] = d0[c];
    } else {
#pragma unroll
      for (int i = 0; i < NS; ++i) {
        S[c][i] = w0[(2 * c * NS + i) * kAdjThreads];
        D[c][i] = w0[((2 * c + 1) * NS + i) * kAdjThreads];
      }
    }
  }
#pragma unroll
  for (int j = 0; j < NS; ++j)
#pragma unroll
    for (int kk = 0; kk < NS; ++kk) yz[j][kk] = S[1][j] * S[2][kk];
  const auto deposit = [&](int j, int kk, double Sx, int64_t o) {
    if (j == 0 && kk == 0) {
#pragma unroll
      for (int c = 0; c < 6; ++c) fx[c] = Sx * fb[c];
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) atomicAdd(a.Fb[c] + o, fx[c] * yz[j][kk]);
  };
  if constexpr (P == 1) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
      grad[c] = Eb[0] * dF[0][c] + Eb[1] * dF[1][c] + Eb[2] * dF[2][c] + Bb[0] * dF[3][c] + Bb[1] * dF[4][c] +
                Bb[2] * dF[5][c];
#pragma unroll
    for (int i = 0; i < NS; ++i) {
      const int64_t ox = (int64_t)((lo[0] + i) & a.mask[0]) * a.Ny;
#pragma unroll
      for (int j = 0; j < NS; ++j) {
        const int64_t oy = (ox + ((lo[1] + j) & a.mask[1])) * a.Nz;
#pragma unroll
        for (int kk = 0; kk < NS; ++kk) deposit(j, kk, S[0][i], oy + ((lo[2] + kk) & a.mask[2]));
      }
    }
  } else {
    node_grad<P, false>(a, lo, S, D, w0, none, grad, [&](int j, int kk, double Sx, int64_t o) {
      double g = fb[0] * __ldg(a.F[0] + o);
#pragma unroll
      for (int c = 1; c < 6; ++c) g = fma(fb[c], __ldg(a.F[c] + o), g);
      deposit(j, kk, Sx, o);
      return g;
    });
  }
  for (int c = 0; c < 3; ++c) xb[c] = fma(a.inv_dx[c], grad[c], xb[c]);
  a.xb[p] = xb[0];
  a.yb[p] = xb[1];
  a.zb[p] = xb[2];
  a.uxb[p] = umb[0];
  a.uyb[p] = umb[1];
  a.uzb[p] = umb[2];
}

// y += x (the two adjoints of rho^{n+1}: from the update and from the caller)
__global__ void add_kernel(double* y, const double* x, int64_t n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    y[e] += x[e];
}

template <class P>
bool nonnull(P const* a, int n) {
  if (!a) return false;
  for (int i = 0; i < n; ++i)
    if (!a[i]) return false;
  return true;
}

#define ADJ_TRY(x)                 \
  do {                             \
    pic_status s_ = (x);           \
    if (s_ != PIC_OK) return s_;   \
  } while (0)

// Yee real arrays -> paper-convention spectra in ctx->EBh (through G)
pic_status to_paper(pic_ctx* ctx, const double* const* F6) {
  CRPtr6 in;
  CPtr6 g;
  for (int c = 0; c < 6; ++c) {
    in.p[c] = F6[c];
    g.p[c] = ctx->G + c * ctx->nmode;
  }
  {
    StageScope t(ctx, STAGE_FFT, 3);
    ADJ_TRY(fft_r2c<double>(ctx, in, g, 6));
  }
  StageScope t(ctx, STAGE_OTHER, 1);
  return psatd_load<double2>(ctx, ctx->G, ctx->EBh);
}

}  // namespace

extern "C" pic_status pic_adjoint_step(pic_ctx* ctx, const double* const E[3], const double* const B[3],
                                       const pic_species* sp, int n_species, double* const Ebar[3],
                                       double* const Bbar[3], double* rhobar, const pic_species_adjoint* spbar) {
  if (!ctx) return PIC_ERR_ARG;
  if (ctx->precision != PIC_FP64) return pic_set_error(ctx, PIC_ERR_ARG, "the adjoint step is FP64 only");
  if (ctx->variant == PIC_PSATD_AVERAGED_GALILEAN)
    return pic_set_error(ctx, PIC_ERR_UNSUPPORTED, "no adjoint for the averaged Galilean variant");
  if (ctx->filter_passes > 0 || ctx->pusher != PIC_PUSHER_BORIS || ctx->cycle != PIC_CYCLE_HYBRID)
    return pic_set_error(ctx, PIC_ERR_UNSUPPORTED,
                         "the adjoint covers the hybrid cycle with the Boris pusher and no smoothing");
  if (!nonnull(E, 3) || !nonnull(B, 3) || !nonnull(Ebar, 3) || !nonnull(Bbar, 3) || !rhobar)
    return pic_set_error(ctx, PIC_ERR_ARG, "null field pointer");
  {
    const void* ptrs[13] = {E[0], E[1], E[2], B[0], B[1], B[2], Ebar[0], Ebar[1], Ebar[2], Bbar[0], Bbar[1], Bbar[2],
                            rhobar};
    PIC_NEED_ALIGNED(ctx, ptrs, 13, 16);
  }
  if (n_species < 0 || (n_species > 0 && (!sp || !spbar))) return pic_set_error(ctx, PIC_ERR_ARG, "species");
  for (int s = 0; s < n_species; ++s) {
    if (sp[s].n != spbar[s].n) return pic_set_error(ctx, PIC_ERR_ARG, "species %d: adjoint size mismatch", s);
    if (sp[s].n > 0 && (!sp[s].x || !sp[s].y || !sp[s].z || !sp[s].ux || !sp[s].uy || !sp[s].uz || !sp[s].w ||
                        !spbar[s].x || !spbar[s].y || !spbar[s].z || !spbar[s].ux || !spbar[s].uy || !spbar[s].uz))
      return pic_set_error(ctx, PIC_ERR_ARG, "species %d: null array", s);
    if (!(sp[s].m > 0.0)) return pic_set_error(ctx, PIC_ERR_ARG, "species %d: mass must be > 0", s);
  }
  const int64_t nc = ctx->ncell, nm = ctx->nmode;
  if (!ctx->adj_work) {
    cudaError_t e = cudaMalloc(&ctx->adj_work, 8 * nc * sizeof(double));
    if (e != cudaSuccess) {
      cudaGetLastError();
      ctx->adj_work = nullptr;
      return pic_set_error(ctx, PIC_ERR_NOMEM, "adjoint work arrays");
    }
  }
  double* rbn = ctx->adj_work;            // rhobar^n
  double* rbp = ctx->adj_work + nc;       // rhobar^{n+1} from the update
  double* fb = ctx->adj_work + 2 * nc;    // [6] nodal force adjoints
  // 1. nodal E, B at t^n (forward recompute): centered in real space (work array: Jn, free until step 2)
  const double* F6[6] = {E[0], E[1], E[2], B[0], B[1], B[2]};
  {
    double* nodal6[6];
    for (int c = 0; c < 6; ++c) nodal6[c] = ctx->nodal + c * nc;
    StageScope t(ctx, STAGE_OTHER, center_launches(ctx, true));
    ADJ_TRY(center_to_nodal(ctx, F6, nodal6));
  }
  // 2. transpose of the update on the incoming field adjoints
  const double* Fb6[6] = {Ebar[0], Ebar[1], Ebar[2], Bbar[0], Bbar[1], Bbar[2]};
  ADJ_TRY(to_paper(ctx, Fb6));
  {
    StageScope t(ctx, STAGE_UPDATE, 1);
    ADJ_TRY(psatd_adjoint_update(ctx, ctx->EBh, ctx->G));
  }
  {
    CPtr6 g;
    RPtr6 o;
    for (int c = 0; c < 5; ++c) g.p[c] = ctx->G + c * nm;
    for (int c = 0; c < 3; ++c) o.p[c] = ctx->Jn + c * nc;   // nodal Jbar
    o.p[3] = rbn;
    o.p[4] = rbp;
    StageScope t(ctx, STAGE_FFT, 3);
    ADJ_TRY(fft_c2r<double>(ctx, g, o, 5));
  }
  {
    StageScope t(ctx, STAGE_OTHER, 1);
    add_kernel<<<(unsigned)std::min<int64_t>((nc + 255) / 256, 152 * 16), 256, 0, ctx->stream>>>(rbp, rhobar, nc);
    PIC_LAUNCH_CHECK(ctx);
  }
  // 3. particles, reversed
  PIC_CUDA_TRY(ctx, cudaMemsetAsync(fb, 0, 6 * nc * sizeof(double), ctx->stream));
  for (int s = 0; s < n_species; ++s) {
    if (sp[s].n == 0) continue;
    AdjArgs a;
    a.x = sp[s].x;
    a.y = sp[s].y;
    a.z = sp[s].z;
    a.ux = sp[s].ux;
    a.uy = sp[s].uy;
    a.uz = sp[s].uz;
    a.w = sp[s].w;
    a.xb = spbar[s].x;
    a.yb = spbar[s].y;
    a.zb = spbar[s].z;
    a.uxb = spbar[s].ux;
    a.uyb = spbar[s].uy;
    a.uzb = spbar[s].uz;
    a.n = sp[s].n;
    for (int c = 0; c < 6; ++c) {
      a.F[c] = ctx->nodal + c * nc;
      a.Fb[c] = fb + c * nc;
    }
    for (int c = 0; c < 3; ++c) a.Jb[c] = ctx->Jn + c * nc;
    a.Rb = rbp;
    for (int d = 0; d < 3; ++d) {
      a.inv_dx[d] = 1.0 / ctx->dx[d];
      a.L[d] = (double)ctx->N[d] * ctx->dx[d];
      a.mask[d] = (int)ctx->N[d] - 1;
      a.vg[d] = ctx->variant == PIC_PSATD_STANDARD ? 0.0 : ctx->vg[d];
    }
    a.Ny = ctx->N[1];
    a.Nz = ctx->N[2];
    a.k = sp[s].q * ctx->dt / (2.0 * sp[s].m);
    a.dt = ctx->dt;
    a.inv_c2 = 1.0 / (ctx->c * ctx->c);
    a.qw_scale = sp[s].q / (ctx->dx[0] * ctx->dx[1] * ctx->dx[2]);
    const int bs = kAdjThreads;
    const unsigned nb = (unsigned)((a.n + bs - 1) / bs);
    StageScope t(ctx, STAGE_PUSH, 1);
    switch (ctx->shape_order) {
      case 1: adjoint_push_kernel<1><<<nb, bs, 0, ctx->stream>>>(a); break;
      case 2: adjoint_push_kernel<2><<<nb, bs, 0, ctx->stream>>>(a); break;
      default: adjoint_push_kernel<3><<<nb, bs, 0, ctx->stream>>>(a); break;
    }
    PIC_LAUNCH_CHECK(ctx);
  }
  // 4. transpose of the E, B centering: EBh += zeta * DFT(force adjoints); back to Yee
  {
    CRPtr6 in;
    CPtr6 g;
    for (int c = 0; c < 6; ++c) {
      in.p[c] = fb + c * nc;
      g.p[c] = ctx->G + c * nm;
    }
    StageScope t(ctx, STAGE_FFT, 3);
    ADJ_TRY(fft_r2c<double>(ctx, in, g, 6));
  }
  {
    StageScope t(ctx, STAGE_OTHER, 1);
    ADJ_TRY(psatd_add_zeta(ctx, ctx->EBh, ctx->G));
  }
  {
    CPtr6 g;
    RPtr6 o;
    for (int c = 0; c < 6; ++c) g.p[c] = ctx->G + c * nm;
    for (int c = 0; c < 3; ++c) {
      o.p[c] = Ebar[c];
      o.p[3 + c] = Bbar[c];
    }
    {
      StageScope t(ctx, STAGE_OTHER, 1);
      ADJ_TRY(psatd_store<double2>(ctx, ctx->EBh, ctx->G));
    }
    StageScope t(ctx, STAGE_FFT, 3);
    ADJ_TRY(fft_c2r<double>(ctx, g, o, 6));
  }
  // 5. adjoint of rho^n
  PIC_CUDA_TRY(ctx, cudaMemcpyAsync(rhobar, rbn, nc * sizeof(double), cudaMemcpyDeviceToDevice, ctx->stream));
  return PIC_OK;
}
