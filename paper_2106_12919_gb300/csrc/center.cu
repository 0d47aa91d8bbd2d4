// Finite-order centering between the nodal and Yee grids as real-space stencils
// (Sec. 3, Eq. staggered_finite_sum, periodic).  Between its steps pic_step applies
// the same operators as their Fourier symbol inside the k-space update; these
// kernels are the stand-alone form of the two centering rows of the step, the
// centering of the fields a call starts from and of the J it returns, and the
// centering of the FDTD cycle (FP64 and FP32), which also filters its J here.
//
// staggered -> nodal along axis a: f_j = sum_n w_n (s[j+n-1] + s[j-n]),
// nodal -> staggered:               f_{j+1/2} = sum_n w_n (g[j+n] + g[j-n+1]),
// with w_n = alpha^s_{m,n} / 2 and s[i] the value at (i + 1/2) dx.
#include "pic_internal.cuh"

namespace {

template <class T>
struct StencilArgs {
  const T* in;
  T* out;
  int ncell;
  int shift, mask;  // the axis: index stride 2^shift, coordinate j = (e >> shift) & mask
  int mode;  // 0: nodal -> staggered, 1: staggered -> nodal, 2: bilinear (1/4, 1/2, 1/4) filter
  int m;
  T w[PIC_MAX_CENTER_M];
};

// One output element per thread; grids are powers of two (at most 2^30 cells), so the index
// arithmetic is 32-bit shifts and masks.
template <class T>
__global__ void __launch_bounds__(256) stencil_kernel(StencilArgs<T> a) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.ncell) return;
  const int j = (e >> a.shift) & a.mask;
  const int base = e - (j << a.shift);
  const T* in = a.in;
  if (a.mode == 2) {
    // f_j <- f_{j-1} / 4 + f_j / 2 + f_{j+1} / 4 (Sec. 2, the smoothing of the deposits)
    a.out[e] = T(0.25) * in[base + (((j - 1) & a.mask) << a.shift)] + T(0.5) * in[e] +
               T(0.25) * in[base + (((j + 1) & a.mask) << a.shift)];
    return;
  }
  // mode 1: f_j = sum_n w_n (s[j+n-1] + s[j-n]); mode 0: f_{j+1/2} = sum_n w_n (g[j+n] + g[j-n+1])
  const int d = a.mode == 1 ? -1 : 0;
  T acc = T(0);
#pragma unroll
  for (int n = 1; n <= PIC_MAX_CENTER_M; ++n) {
    if (n > a.m) break;
    const int i1 = (j + n + d) & a.mask, i2 = (j - n + 1 + d) & a.mask;
    acc += a.w[n - 1] * (in[base + (i1 << a.shift)] + in[base + (i2 << a.shift)]);
  }
  a.out[e] = acc;
}

// The centering stencils of m <= 8 on large grids: a thread forms several consecutive outputs of a line
// from one register window (R + 2m - 1 loads for R outputs, where one output per thread takes 2m).  The
// field is a few L2-resident arrays, so the loads through L1 bound these passes, not HBM: 4.2 million
// FP32 cells, m = 8 along z and 4 transverse, the 12 passes of a step 0.42 -> 0.22 ms.
//
// x and y: 8 outputs along the axis, lanes along z.  off: first input of output j is j - M + off.
template <class T, int M>
__global__ void __launch_bounds__(256) stencil_line_kernel(StencilArgs<T> a, int off) {
  constexpr int R = 8;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.ncell / R) return;
  // t = (outer, block of 8 along the axis, inner of 2^shift elements)
  const int inner = t & ((1 << a.shift) - 1), q = t >> a.shift;
  const int nb = (a.mask + 1) / R, j0 = (q & (nb - 1)) * R, outer = q / nb;
  const int base = ((outer * (a.mask + 1)) << a.shift) + inner;
  const T* in = a.in + base;
  T v[R + 2 * M - 1];
#pragma unroll
  for (int i = 0; i < R + 2 * M - 1; ++i) v[i] = in[((j0 - M + off + i) & a.mask) << a.shift];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    T acc = T(0);
#pragma unroll
    for (int n = 1; n <= M; ++n) acc += a.w[n - 1] * (v[r + M + n - 1] + v[r + M - n]);
    a.out[base + ((j0 + r) << a.shift)] = acc;
  }
}

// z: 4 outputs from 16-byte loads (V elements); OFF as off above
template <class T, int M, int OFF>
__global__ void __launch_bounds__(256) stencil_z_kernel(StencilArgs<T> a) {
  constexpr int R = 4, V = 16 / (int)sizeof(T);
  constexpr int LO = (M - OFF + V - 1) / V * V;        // window start before the first output, aligned
  constexpr int NV = (LO + R - 1 + M - 1 + OFF) / V + 1;
  struct alignas(16) Vec { T v[V]; };
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.ncell / R) return;
  const int e = t * R, z0 = e & a.mask, base = e - z0;
  T v[NV * V];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const Vec x = *reinterpret_cast<const Vec*>(a.in + base + ((z0 - LO + i * V) & a.mask));
#pragma unroll
    for (int q = 0; q < V; ++q) v[i * V + q] = x.v[q];
  }
  constexpr int S = LO - (M - OFF);  // first input of output 0 in the window
  T o[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    o[r] = T(0);
#pragma unroll
    for (int n = 1; n <= M; ++n) o[r] += a.w[n - 1] * (v[S + r + M + n - 1] + v[S + r + M - n]);
  }
#pragma unroll
  for (int i = 0; i < R / V; ++i) {
    Vec x;
#pragma unroll
    for (int q = 0; q < V; ++q) x.v[q] = o[i * V + q];
    *reinterpret_cast<Vec*>(a.out + e + i * V) = x;
  }
}

template <class T, int M>
void launch_window(const StencilArgs<T>& s, int axis, cudaStream_t st) {
  const int off = s.mode == 1 ? 0 : 1;
  if (axis == 2) {
    const unsigned nb = (unsigned)((s.ncell / 4 + 255) / 256);
    if (off) stencil_z_kernel<T, M, 1><<<nb, 256, 0, st>>>(s);
    else stencil_z_kernel<T, M, 0><<<nb, 256, 0, st>>>(s);
  } else {
    stencil_line_kernel<T, M><<<(unsigned)((s.ncell / 8 + 255) / 256), 256, 0, st>>>(s, off);
  }
}

// true when a window kernel ran: below 2^20 cells their fewer threads leave SMs idle, and unaligned
// arrays cannot take the 16-byte loads
constexpr int64_t kWindowCells = int64_t(1) << 20;
template <class T>
bool launch_window_m(const StencilArgs<T>& s, int axis, cudaStream_t st) {
  if (s.mode == 2 || s.ncell < kWindowCells) return false;
  if (axis == 2 && (reinterpret_cast<uintptr_t>(s.in) | reinterpret_cast<uintptr_t>(s.out)) % 16 != 0) return false;
  switch (s.m) {
    case 1: launch_window<T, 1>(s, axis, st); return true;
    case 2: launch_window<T, 2>(s, axis, st); return true;
    case 3: launch_window<T, 3>(s, axis, st); return true;
    case 4: launch_window<T, 4>(s, axis, st); return true;
    case 5: launch_window<T, 5>(s, axis, st); return true;
    case 6: launch_window<T, 6>(s, axis, st); return true;
    case 7: launch_window<T, 7>(s, axis, st); return true;
    case 8: launch_window<T, 8>(s, axis, st); return true;
  }
  return false;
}

int lg2i(int64_t n) {
  int s = 0;
  while ((int64_t(1) << s) < n) ++s;
  return s;
}

template <class T>
pic_status run(pic_ctx* ctx, const T* in, T* out, int axis, int mode) {
  StencilArgs<T> s;
  memset(&s, 0, sizeof(s));
  s.in = in;
  s.out = out;
  s.ncell = (int)ctx->ncell;
  s.shift = axis == 0 ? lg2i(ctx->N[1]) + lg2i(ctx->N[2]) : axis == 1 ? lg2i(ctx->N[2]) : 0;
  s.mask = (int)ctx->N[axis] - 1;
  s.mode = mode;
  s.m = ctx->cw[axis].m;
  for (int n = 0; n < s.m; ++n) s.w[n] = (T)ctx->cw[axis].w[n];
  const int bs = 256;
  if (launch_window_m(s, axis, ctx->stream)) {
    PIC_LAUNCH_CHECK(ctx);
    return PIC_OK;
  }
  stencil_kernel<T><<<(unsigned)((ctx->ncell + bs - 1) / bs), bs, 0, ctx->stream>>>(s);
  PIC_LAUNCH_CHECK(ctx);
  return PIC_OK;
}

// staggered axes of E^x..B^z as bit masks (x = 1, y = 2, z = 4)
const int kStag[6] = {1, 2, 4, 2 | 4, 1 | 4, 1 | 2};

// Apply the stencils of every axis in mask (x, y, z order) from in to out,
// using two work arrays for the intermediate results.
template <class T>
pic_status apply(pic_ctx* ctx, const T* in, T* out, int mask, int mode, T* w0, T* w1) {
  int axes[3], na = 0;
  for (int a = 0; a < 3; ++a)
    if (mask & (1 << a)) axes[na++] = a;
  const T* src = in;
  for (int q = 0; q < na; ++q) {
    T* dst = (q == na - 1) ? out : (q % 2 == 0 ? w0 : w1);
    PIC_TRY(run<T>(ctx, src, dst, axes[q], mode));
    src = dst;
  }
  return PIC_OK;
}

// Small grids: one pass along its own axis for each of up to six components in one launch (launches
// are most of their time).
template <class T>
struct BatchArgs {
  const T* in[6];
  T* out[6];
  int axis[6];
  int shift[3], mask[3], m[3];
  T w[3][PIC_MAX_CENTER_M];
  int ncell, mode;
};

template <class T>
__global__ void __launch_bounds__(256) stencil_batch_kernel(BatchArgs<T> a) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.ncell) return;
  const int c = blockIdx.y, x = a.axis[c];
  const int shift = a.shift[x], mask = a.mask[x], j = (e >> shift) & mask;
  const T* in = a.in[c] + (e - (j << shift));
  const int d = a.mode == 1 ? -1 : 0;
  T acc = T(0);
#pragma unroll 4
  for (int n = 1; n <= a.m[x]; ++n)
    acc += a.w[x][n - 1] * (in[((j + n + d) & mask) << shift] + in[((j - n + 1 + d) & mask) << shift]);
  a.out[c][e] = acc;
}

template <class T>
pic_status run_batch(pic_ctx* ctx, const T* const* in, T* const* out, const int* axis, int n, int mode) {
  BatchArgs<T> b;
  memset(&b, 0, sizeof(b));
  for (int c = 0; c < n; ++c) {
    b.in[c] = in[c];
    b.out[c] = out[c];
    b.axis[c] = axis[c];
  }
  b.shift[1] = lg2i(ctx->N[2]);
  b.shift[0] = b.shift[1] + lg2i(ctx->N[1]);
  for (int x = 0; x < 3; ++x) {
    b.mask[x] = (int)ctx->N[x] - 1;
    b.m[x] = ctx->cw[x].m;
    for (int k = 0; k < b.m[x]; ++k) b.w[x][k] = (T)ctx->cw[x].w[k];
  }
  b.ncell = (int)ctx->ncell;
  b.mode = mode;
  stencil_batch_kernel<T><<<dim3((unsigned)((ctx->ncell + 255) / 256), n), 256, 0, ctx->stream>>>(b);
  PIC_LAUNCH_CHECK(ctx);
  return PIC_OK;
}

}  // namespace

int center_launches(const pic_ctx* ctx, bool to_nodal) {
  return ctx->ncell < kWindowCells ? (to_nodal ? 2 : 1) : (to_nodal ? 9 : 3);
}

template <class T>
pic_status center_to_nodal_t(pic_ctx* ctx, const T* const F[6], T* const out[6], T* w) {
  const int64_t nc = ctx->ncell;
  if (nc < kWindowCells) {
    // E^x, E^y, E^z along their axis; B^x along y, B^y and B^z along x into w, then along z, z, y
    T* const first[6] = {out[0], out[1], out[2], w, w + nc, w + 2 * nc};
    const T* const second[3] = {w, w + nc, w + 2 * nc};
    const int ax1[6] = {0, 1, 2, 1, 0, 0}, ax2[3] = {2, 2, 1};
    PIC_TRY(run_batch<T>(ctx, F, first, ax1, 6, 1));
    return run_batch<T>(ctx, second, out + 3, ax2, 3, 1);
  }
  for (int c = 0; c < 6; ++c) PIC_TRY(apply<T>(ctx, F[c], out[c], kStag[c], 1, w, w + nc));
  return PIC_OK;
}

template <class T>
pic_status center_to_yee_t(pic_ctx* ctx, const T* const Jn[3], T* const out[3]) {
  if (ctx->ncell < kWindowCells) {
    const int ax[3] = {0, 1, 2};
    return run_batch<T>(ctx, Jn, out, ax, 3, 0);
  }
  for (int c = 0; c < 3; ++c) PIC_TRY(apply<T>(ctx, Jn[c], out[c], kStag[c], 0, (T*)nullptr, (T*)nullptr));
  return PIC_OK;
}

template <class T>
pic_status bilinear_filter_t(pic_ctx* ctx, T* f, int passes, T* w0, T* w1) {
  for (int p = 0; p < passes; ++p) {
    PIC_TRY(run<T>(ctx, f, w0, 0, 2));
    PIC_TRY(run<T>(ctx, w0, w1, 1, 2));
    PIC_TRY(run<T>(ctx, w1, f, 2, 2));
  }
  return PIC_OK;
}

template pic_status center_to_nodal_t<double>(pic_ctx*, const double* const[6], double* const[6], double*);
template pic_status center_to_nodal_t<float>(pic_ctx*, const float* const[6], float* const[6], float*);
template pic_status center_to_yee_t<double>(pic_ctx*, const double* const[3], double* const[3]);
template pic_status center_to_yee_t<float>(pic_ctx*, const float* const[3], float* const[3]);
template pic_status bilinear_filter_t<double>(pic_ctx*, double*, int, double*, double*);
template pic_status bilinear_filter_t<float>(pic_ctx*, float*, int, float*, float*);

pic_status center_to_nodal(pic_ctx* ctx, const double* const F[6], double* const out[6]) {
  return center_to_nodal_t<double>(ctx, F, out, ctx->Jn);
}

pic_status center_to_yee(pic_ctx* ctx, const double* const Jn[3], double* const out[3]) {
  return center_to_yee_t<double>(ctx, Jn, out);
}
