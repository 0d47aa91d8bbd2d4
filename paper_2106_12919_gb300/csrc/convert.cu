// Conversions between the FP64 and FP32 particle representations, and the adjoint seed of the
// probe-box field energy (the loss of the reverse mode).
//
// FP32-form positions: each coordinate is an integer cell i and an FP32 offset f in [0, 1) with
// x = (i + f) dx.  The split takes t = x * (1/dx) rounded to FP64 (the multiply of the FP64
// form's nearest-node rule), i = floor(t), f = t - i (exact in FP64) rounded once to FP32; an
// offset that rounds to 1.0 moves the particle to offset 0 of the next cell, and the cell wraps
// into [0, N).  The join is x = (i + f) * dx in FP64 (i + f is exact).  Products use __dmul_rn so
// that no multiply is contracted into an FMA: the results are the correctly rounded ones.
#include "pic_internal.cuh"

namespace {

struct SplitArgs {
  const double* x[3];
  const double* u[3];
  const double* w;
  const int64_t* id_in;
  int32_t* cell;
  float* f[3];
  float* u32[3];
  float* w32;
  int64_t* id_out;
  double inv_dx[3];
  int mask[3];  // N - 1 (powers of two)
  int sy, sz;   // log2 of Ny, Nz
  int64_t n;
};

// Both kernels move 104 bytes per particle, 15.5 ps at the copy bandwidth.  They were bound by the FP64
// pipe: floors, additions and conversions between formats, at 1.7 to 2 per clock and SM, took 34 (split) and
// 32 ps (join, 68.1 million particles).  On the bit patterns, with one FP64 product per coordinate left,
// 19.5 and 20.9 ps (16.8 million).

// (float)v, rounded to nearest even: normal results and zeros without the FP64 pipe
__device__ __forceinline__ float narrow(double v) {
  const uint64_t b = (uint64_t)__double_as_longlong(v), m = b & 0x7fffffffffffffffull;
  const uint32_t sign = (uint32_t)(b >> 63) << 31;
  if (m == 0ull) return __uint_as_float(sign);
  if ((uint32_t)(m >> 52) - 897u >= 253u) return __double2float_rn(v);  // (the result's exponent field: 1 .. 253)
  const uint64_t r = m - (896ull << 52);
  return __uint_as_float((uint32_t)((r + 0x0fffffffull + ((r >> 29) & 1ull)) >> 29) | sign);
}

// cell (not wrapped) and offset of t = x / dx: floor(t), and t - floor(t) rounded to FP32
__device__ __forceinline__ int split_cell(double t, float& f) {
  const uint64_t b = (uint64_t)__double_as_longlong(t);
  const int sh = 1075 - (int)(b >> 52);                      // t = m 2^-sh
  const uint64_t m = (b & 0xfffffffffffffull) | (1ull << 52);
  const int i = sh > 52 ? 0 : (int)(m >> (sh & 63));
  const uint64_t r = sh > 52 ? m : m & ((1ull << (sh & 63)) - 1ull);
  const int lz = __clzll((long long)r), ef = 190 - lz - sh;  // the offset's exponent field
  // t < 0, t >= 2^31 or not finite (sh < 22, the sign being part of it); tiny or zero offsets
  if (sh < 22 || ef < 1 || r == 0ull) {
    if (sh >= 22 && r == 0ull) {
      f = 0.0f;
      return i;
    }
    const double c = floor(t);
    f = __double2float_rn(t - c);
    return (int)(int64_t)c;
  }
  const uint64_t n = r << lz;
  const uint32_t m24 = (uint32_t)(n >> 40);
  const uint64_t rest = n << 24;
  const uint32_t up = rest > (1ull << 63) || (rest == (1ull << 63) && (m24 & 1u)) ? 1u : 0u;
  f = __uint_as_float(((uint32_t)ef << 23) + (m24 & 0x7fffffu) + up);
  return i;
}

__global__ void split_kernel(SplitArgs a) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < a.n; p += (int64_t)gridDim.x * blockDim.x) {
    int idx[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      float f;
      int i = split_cell(__dmul_rn(a.x[d][p], a.inv_dx[d]), f);
      if (f == 1.0f) f = 0.0f, ++i;
      idx[d] = i & a.mask[d];
      a.f[d][p] = f;
      a.u32[d][p] = narrow(a.u[d][p]);
    }
    a.cell[p] = (((idx[0] << a.sy) + idx[1]) << a.sz) + idx[2];
    a.w32[p] = narrow(a.w[p]);
    if (a.id_out) a.id_out[p] = a.id_in[p];
  }
}

struct JoinArgs {
  const int32_t* cell;
  const float* f[3];
  const float* u32[3];
  const float* w32;
  const int64_t* id_in;
  double* x[3];
  double* u[3];
  double* w;
  int64_t* id_out;
  double dx[3];
  int mask[3];  // N - 1 (powers of two)
  int sy, sz;   // log2 of Ny, Nz
  int64_t n;
};

// (double)f, exact, without the FP64 pipe for normal numbers
__device__ __forceinline__ double widen(float f) {
  const uint32_t b = __float_as_uint(f);
  if (((b >> 23) & 0xffu) - 1u >= 254u) return (double)f;  // zero, subnormal, infinite, NaN
  const uint64_t m = ((uint64_t)(b & 0x7fffffffu) << 29) + ((uint64_t)(1023 - 127) << 52);
  return __longlong_as_double((int64_t)(m | ((uint64_t)(b >> 31) << 63)));
}

// i + f for a cell 0 <= i < 1024 and an offset f in [0, 1): exact and without the FP64 pipe from f = 2^-20
// (the sum's lowest bit is then 53 or fewer below its highest) and for f = 0
__device__ __forceinline__ double cell_plus(int i, float f) {
  const uint32_t b = __float_as_uint(f), e = b >> 23;
  if ((uint32_t)i >= 1024u || (b != 0u && e - 107u >= 20u)) return (double)i + widen(f);
  const uint64_t s = ((uint64_t)(uint32_t)i << 52) +
                     (b == 0u ? 0ull : (uint64_t)((b & 0x7fffffu) | 0x800000u) << (e - 98u & 63u));
  if (s == 0ull) return 0.0;
  const int lz = __clzll((long long)s);
  return __longlong_as_double((int64_t)(((uint64_t)(1034 - lz) << 52) | (s << lz << 1 >> 12)));
}

__global__ void join_kernel(JoinArgs a) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < a.n; p += (int64_t)gridDim.x * blockDim.x) {
    const int c = a.cell[p];
    const int idx[3] = {c >> (a.sy + a.sz), (c >> a.sz) & a.mask[1], c & a.mask[2]};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      a.x[d][p] = __dmul_rn(cell_plus(idx[d], a.f[d][p]), a.dx[d]);
      a.u[d][p] = widen(a.u32[d][p]);
    }
    a.w[p] = widen(a.w32[p]);
    if (a.id_out) a.id_out[p] = a.id_in[p];
  }
}

struct SeedArgs {
  const double* E[3];
  const double* B[3];
  double* Eb[3];
  double* Bb[3];
  int64_t lo[3], hi[3];
  int64_t N[3];
  int64_t ncell;
  double se, sb;
};

// Ebar = se E, Bbar = sb B on the cells of the box [lo, hi), 0 elsewhere.
__global__ void energy_seed_kernel(SeedArgs a) {
  for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < a.ncell;
       m += (int64_t)gridDim.x * blockDim.x) {
    const int64_t iz = m % a.N[2], r = m / a.N[2];
    const int64_t iy = r % a.N[1], ix = r / a.N[1];
    const bool in = ix >= a.lo[0] && ix < a.hi[0] && iy >= a.lo[1] && iy < a.hi[1] && iz >= a.lo[2] &&
                    iz < a.hi[2];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      a.Eb[c][m] = in ? a.se * a.E[c][m] : 0.0;
      a.Bb[c][m] = in ? a.sb * a.B[c][m] : 0.0;
    }
  }
}

int grid_blocks(int64_t n) {
  const int64_t b = (n + 255) / 256;
  return (int)(b < 152 * 16 ? (b > 0 ? b : 1) : 152 * 16);
}

pic_status species_pair_check(pic_ctx* ctx, const pic_species* s64, const pic_species32* s32) {
  if (!s64 || !s32) return pic_set_error(ctx, PIC_ERR_ARG, "null species");
  if (s64->n < 0 || s64->n != s32->n) return pic_set_error(ctx, PIC_ERR_ARG, "species counts differ or are negative");
  if (s64->n > ((int64_t)1 << 31) - 1) return pic_set_error(ctx, PIC_ERR_CAPACITY, "more than 2^31-1 particles");
  if (s64->n == 0) return PIC_OK;
  if (!s64->x || !s64->y || !s64->z || !s64->ux || !s64->uy || !s64->uz || !s64->w)
    return pic_set_error(ctx, PIC_ERR_ARG, "null FP64 species array");
  if (!s32->cell || !s32->fx || !s32->fy || !s32->fz || !s32->ux || !s32->uy || !s32->uz || !s32->w)
    return pic_set_error(ctx, PIC_ERR_ARG, "null FP32 species array");
  if ((s64->id == nullptr) != (s32->id == nullptr))
    return pic_set_error(ctx, PIC_ERR_ARG, "id given on one side only");
  return PIC_OK;
}

}  // namespace

extern "C" {

pic_status pic_species32_from_species(pic_ctx* ctx, const pic_species* in, const pic_species32* out) {
  if (!ctx) return PIC_ERR_ARG;
  PIC_TRY(species_pair_check(ctx, in, out));
  if (in->n == 0) return PIC_OK;
  SplitArgs a;
  a.x[0] = in->x;
  a.x[1] = in->y;
  a.x[2] = in->z;
  a.u[0] = in->ux;
  a.u[1] = in->uy;
  a.u[2] = in->uz;
  a.w = in->w;
  a.id_in = in->id;
  a.cell = out->cell;
  a.f[0] = out->fx;
  a.f[1] = out->fy;
  a.f[2] = out->fz;
  a.u32[0] = out->ux;
  a.u32[1] = out->uy;
  a.u32[2] = out->uz;
  a.w32 = out->w;
  a.id_out = out->id;
  for (int d = 0; d < 3; ++d) {
    a.inv_dx[d] = 1.0 / ctx->dx[d];
    a.mask[d] = (int)ctx->N[d] - 1;
  }
  a.sy = __builtin_ctzll((unsigned long long)ctx->N[1]);
  a.sz = __builtin_ctzll((unsigned long long)ctx->N[2]);
  a.n = in->n;
  {
    StageScope t(ctx, STAGE_OTHER, 1);
    split_kernel<<<grid_blocks(a.n), 256, 0, ctx->stream>>>(a);
  }
  PIC_LAUNCH_CHECK(ctx);
  return PIC_OK;
}

pic_status pic_species32_to_species(pic_ctx* ctx, const pic_species32* in, const pic_species* out) {
  if (!ctx) return PIC_ERR_ARG;
  PIC_TRY(species_pair_check(ctx, out, in));
  if (in->n == 0) return PIC_OK;
  JoinArgs a;
  a.cell = in->cell;
  a.f[0] = in->fx;
  a.f[1] = in->fy;
  a.f[2] = in->fz;
  a.u32[0] = in->ux;
  a.u32[1] = in->uy;
  a.u32[2] = in->uz;
  a.w32 = in->w;
  a.id_in = in->id;
  a.x[0] = out->x;
  a.x[1] = out->y;
  a.x[2] = out->z;
  a.u[0] = out->ux;
  a.u[1] = out->uy;
  a.u[2] = out->uz;
  a.w = out->w;
  a.id_out = out->id;
  for (int d = 0; d < 3; ++d) {
    a.dx[d] = ctx->dx[d];
    a.mask[d] = (int)ctx->N[d] - 1;
  }
  a.sy = __builtin_ctzll((unsigned long long)ctx->N[1]);
  a.sz = __builtin_ctzll((unsigned long long)ctx->N[2]);
  a.n = in->n;
  {
    StageScope t(ctx, STAGE_OTHER, 1);
    join_kernel<<<grid_blocks(a.n), 256, 0, ctx->stream>>>(a);
  }
  PIC_LAUNCH_CHECK(ctx);
  return PIC_OK;
}

pic_status pic_field_energy_adjoint(pic_ctx* ctx, const double* const E[3], const double* const B[3],
                                    const int64_t box_lo[3], const int64_t box_hi[3], double scale,
                                    double* const Ebar[3], double* const Bbar[3]) {
  if (!ctx) return PIC_ERR_ARG;
  if (ctx->precision != PIC_FP64) return pic_set_error(ctx, PIC_ERR_ARG, "pic_field_energy_adjoint needs an FP64 context");
  if (!E || !B || !Ebar || !Bbar) return pic_set_error(ctx, PIC_ERR_ARG, "null argument");
  for (int c = 0; c < 3; ++c)
    if (!E[c] || !B[c] || !Ebar[c] || !Bbar[c]) return pic_set_error(ctx, PIC_ERR_ARG, "null field pointer");
  if ((box_lo == nullptr) != (box_hi == nullptr)) return pic_set_error(ctx, PIC_ERR_ARG, "give both box corners or neither");
  SeedArgs a;
  for (int d = 0; d < 3; ++d) {
    a.lo[d] = 0;
    a.hi[d] = ctx->N[d];
    a.N[d] = ctx->N[d];
    if (box_lo) {
      if (box_lo[d] < 0 || box_hi[d] > ctx->N[d] || box_lo[d] > box_hi[d])
        return pic_set_error(ctx, PIC_ERR_ARG, "box out of range");
      a.lo[d] = box_lo[d];
      a.hi[d] = box_hi[d];
    }
  }
  for (int c = 0; c < 3; ++c) {
    a.E[c] = E[c];
    a.B[c] = B[c];
    a.Eb[c] = Ebar[c];
    a.Bb[c] = Bbar[c];
  }
  a.ncell = ctx->ncell;
  // W = 1/2 sum (eps0 |E|^2 + |B|^2 / mu0) dV with 1 / mu0 = eps0 c^2
  const double dV = ctx->dx[0] * ctx->dx[1] * ctx->dx[2];
  a.se = scale * ctx->eps0 * dV;
  a.sb = scale * ctx->eps0 * ctx->c * ctx->c * dV;
  {
    StageScope t(ctx, STAGE_OTHER, 1);
    energy_seed_kernel<<<grid_blocks(a.ncell), 256, 0, ctx->stream>>>(a);
  }
  PIC_LAUNCH_CHECK(ctx);
  return PIC_OK;
}

}  // extern "C"
