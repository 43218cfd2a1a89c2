// a3 mass assignment (eq:delgrid, Sec. 2.3) on the grid and on the grid shifted by H/2 (Sec. 3.1).
//
// k_assign_direct: one thread per particle, FP64 weights, FP64 global atomics straight into the grid.
// This is the plain FP64 path (oracle-parity mode and the baseline the fast path is measured
// against): it accepts particles in any order. The FP32 and PK_FIXED64 paths run on the tiled kernels
// of assign_tiles.cu; this file also holds the conversions and weight sums they share.
#include "internal.cuh"

namespace pk {

PK_ERR_ACCESSOR(take_err_assign)

// ---- plain FP64 path ------------------------------------------------------------------------------

template <int P, typename G>
__device__ __forceinline__ void scatter_direct(G* __restrict__ g, const int* c, const double* f, double wgt, int ng,
                                               int ldz) {
  double wx[P], wy[P], wz[P];
  const int sx = bspline<P>(f[0], wx), sy = bspline<P>(f[1], wy), sz = bspline<P>(f[2], wz);
#pragma unroll
  for (int a = 0; a < P; ++a) {
    const int gx = wrap(c[0] + sx + a, ng);
#pragma unroll
    for (int b = 0; b < P; ++b) {
      const int gy = wrap(c[1] + sy + b, ng);
      const double wxy = wgt * wx[a] * wy[b];
      G* row = g + (int64_t(gx) * ng + gy) * ldz;
#pragma unroll
      for (int d = 0; d < P; ++d) atomicAdd(row + wrap(c[2] + sz + d, ng), G(wxy * wz[d]));
    }
  }
}

// The products of the weights by integer instructions. This GPU executes two FP64 operations per clock and SM, and
// the p^3 products per particle and grid held that pipe 83 % busy (L2, which does the atomics, 40 %): a product of
// two 53-bit significands is a few 32-bit multiplies, its exponent an addition. 64 bits are kept between the
// factors (instead of 53) and the node's value is rounded once to the nearest double.
// 128^3 particles on N = 128, PCS, two grids: 1188 us with FP64 products, 744 us so (three
// blocks an SM; with the two that 110 registers leave room for, 760). What is left on the FP64 pipe are the weights.
struct Sig {  // m 2^(e - 63), bit 63 of m set
  uint64_t m;
  int e;
};
__device__ __forceinline__ Sig significand(double w) {  // |w|, normal
  return {(uint64_t(__double_as_longlong(w)) << 11) | 0x8000000000000000ull, ((__double2hiint(w) >> 20) & 0x7ff) - 1023};
}
__device__ __forceinline__ Sig sig_mul(Sig a, Sig b) {
  const uint64_t h = __umul64hi(a.m, b.m);  // in [2^62, 2^64)
  const bool top = int64_t(h) < 0;
  return {top ? h : h << 1, a.e + b.e + (top ? 1 : 0)};
}
// sign * a * b, rounded to nearest; the exponent stays within the normal range (products_fit)
__device__ __forceinline__ double sig_product(Sig a, Sig b, unsigned sign) {
  const Sig p = sig_mul(a, b);
  const uint64_t r = (p.m >> 11) + ((p.m >> 10) & 1u);  // [2^52, 2^53]: bit 52 adds one to the exponent
  return __longlong_as_double((long long)(r + (uint64_t(sign | unsigned(p.e + 1022) << 20) << 32)));
}
// Whether a particle's products run on integers: every factor finite and at least 2^-200 (a float weight below 2^128),
// so that no product leaves the normal range. A stencil's end weight that is zero (f = 0) or tiny goes the FP64 way.
template <int P>
__device__ __forceinline__ bool products_fit(const double* wx, const double* wy, const double* wz, double wgt) {
  constexpr int kMin = (1023 - 200) << 20, kSpan = 400 << 20;
  bool ok = unsigned((__double2hiint(wgt) & 0x7fffffff) - kMin) < unsigned(kSpan);
#pragma unroll
  for (int a = 0; a < P; ++a)
    ok = ok && __double2hiint(wx[a]) >= kMin && __double2hiint(wy[a]) >= kMin && __double2hiint(wz[a]) >= kMin;
  return ok;
}

template <int P>
__device__ __forceinline__ void scatter_products(double* __restrict__ g, const int* c, const double* f, double wgt, int ng,
                                                 int ldz) {
  double wx[P], wy[P], wz[P];
  const int sx = bspline<P>(f[0], wx), sy = bspline<P>(f[1], wy), sz = bspline<P>(f[2], wz);
  if (!products_fit<P>(wx, wy, wz, wgt)) {
    scatter_direct<P>(g, c, f, wgt, ng, ldz);
    return;
  }
  const unsigned sign = unsigned(__double2hiint(wgt)) & 0x80000000u;
  const Sig mw = significand(wgt);
  Sig my[P], mz[P];
  int gz[P];
#pragma unroll
  for (int d = 0; d < P; ++d) {
    my[d] = significand(wy[d]);
    mz[d] = significand(wz[d]);
    gz[d] = wrap(c[2] + sz + d, ng);
  }
#pragma unroll
  for (int a = 0; a < P; ++a) {
    const int gx = wrap(c[0] + sx + a, ng);
    Sig mx = significand(wx[a]);
    if (wgt != 1.0) mx = sig_mul(mx, mw);
#pragma unroll
    for (int b = 0; b < P; ++b) {
      const Sig mxy = sig_mul(mx, my[b]);
      double* row = g + (int64_t(gx) * ng + wrap(c[1] + sy + b, ng)) * ldz;
#pragma unroll
      for (int d = 0; d < P; ++d) atomicAdd(row + gz[d], sig_product(mxy, mz[d], sign));
    }
  }
}

template <int P>
__device__ __forceinline__ void scatter(double* __restrict__ g, const int* c, const double* f, double wgt, int ng, int ldz) {
  if constexpr (P == 1)
    scatter_direct<P>(g, c, f, wgt, ng, ldz);
  else
    scatter_products<P>(g, c, f, wgt, ng, ldz);
}

template <int P, typename G>
__global__ void __launch_bounds__(256, P <= 4 ? 3 : 2) k_assign_direct(const void* __restrict__ pos, int fmt, const float* __restrict__ w, int64_t n, int ng,
                                double box, int interlace, G* __restrict__ g1, G* __restrict__ g2, int ldz) {
  const double scale = double(ng) / box;
  for (int64_t i = gtid(); i < n; i += gstride()) {
    int c[3];
    double f[3];
    if (fmt == PK_POS_F64_XYZ) {
      const double* p = static_cast<const double*>(pos) + 3 * i;
      bool bad = false;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        double x = p[a];
        if (!isfinite(x)) { bad = true; x = 0.0; }
        if (!(x >= 0.0 && x < box)) {  // another periodic image (fmod is the identity on [0, L))
          x = fmod(x, box);
          if (x < 0.0) x += box;
        }
        const double u = x * scale;
        const double fl = floor(u);
        int ci = int(fl);
        f[a] = u - fl;
        if (ci >= ng) ci -= ng;
        c[a] = ci;
      }
      if (bad) { raise_err(PK_DERR_NONFINITE); continue; }
    } else {
      const pk_cellpos r = static_cast<const pk_cellpos*>(pos)[i];
      c[0] = cell_x(r.cell); c[1] = cell_y(r.cell); c[2] = cell_z(r.cell);
      f[0] = r.fx; f[1] = r.fy; f[2] = r.fz;
      if (c[0] >= ng || c[1] >= ng || c[2] >= ng || !(f[0] >= 0.0 && f[0] < 1.0 && f[1] >= 0.0 && f[1] < 1.0 &&
                                                      f[2] >= 0.0 && f[2] < 1.0)) {
        raise_err(PK_DERR_CELLRANGE);
        continue;
      }
    }
    const double wgt = w ? double(w[i]) : 1.0;
    scatter<P>(g1, c, f, wgt, ng, ldz);
    if (interlace) {
      int c2[3];
      double f2[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) c2[a] = c[a] + half_shift(f[a], &f2[a]);
      scatter<P>(g2, c2, f2, wgt, ng, ldz);
    }
  }
}

template <typename G>
static cudaError_t launch_direct(int order, const void* pos, int fmt, const float* w, int64_t n, int ng, double box,
                                 bool interlace, G* g1, G* g2, int ldz, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int threads = 256;
  const int blocks = int(std::min<int64_t>((n + threads - 1) / threads, int64_t(num_sms()) * 16));
  switch (order) {
    case 1: k_assign_direct<1, G><<<blocks, threads, 0, s>>>(pos, fmt, w, n, ng, box, interlace, g1, g2, ldz); break;
    case 2: k_assign_direct<2, G><<<blocks, threads, 0, s>>>(pos, fmt, w, n, ng, box, interlace, g1, g2, ldz); break;
    case 3: k_assign_direct<3, G><<<blocks, threads, 0, s>>>(pos, fmt, w, n, ng, box, interlace, g1, g2, ldz); break;
    case 4: k_assign_direct<4, G><<<blocks, threads, 0, s>>>(pos, fmt, w, n, ng, box, interlace, g1, g2, ldz); break;
    case 5: k_assign_direct<5, G><<<blocks, threads, 0, s>>>(pos, fmt, w, n, ng, box, interlace, g1, g2, ldz); break;
    case 6: k_assign_direct<6, G><<<blocks, threads, 0, s>>>(pos, fmt, w, n, ng, box, interlace, g1, g2, ldz); break;
    default: return cudaErrorInvalidValue;
  }
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_assign_direct_f64(int order, const void* pos, int fmt, const float* w, int64_t n, int ng, double box,
                                     bool interlace, double* g1, double* g2, int ldz, cudaStream_t s) {
  return launch_direct<double>(order, pos, fmt, w, n, ng, box, interlace, g1, g2, ldz, s);
}

// ---- small helpers ---------------------------------------------------------------------------------

// v 2^-F rounded to the nearest double (ties to even), as double(v) times a power of two gives it, by integer
// instructions: conversions run on the FP64 pipe.
__device__ __forceinline__ double fixed_value(long long v, int F) {
  const unsigned long long mag = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  if (mag == 0) return 0.0;
  const int lz = __clzll((long long)mag);
  const unsigned long long m = mag << lz;  // bit 63 set
  unsigned long long r = m >> 11;
  const unsigned rest = unsigned(m) & 0x7ffu;
  r += rest > 0x400u || (rest == 0x400u && (r & 1u)) ? 1u : 0u;  // [2^52, 2^53]: bit 52 adds one to the exponent
  const unsigned long long sign = v < 0 ? 0x8000000000000000ull : 0ull;
  return __longlong_as_double((long long)(r + ((unsigned long long)(1022 + 63 - lz - F) << 52) | sign));
}

// In place, both grids (g2 may be null). F costs an FP64 logarithm, which one thread of a block takes: in every thread it
// took 27 of 35 us per grid of 2.1 M nodes (FP64 runs at two operations per clock and SM); both grids 17 us so.
__global__ void __launch_bounds__(256) k_fixed_to_double(unsigned long long* __restrict__ g1, unsigned long long* __restrict__ g2,
                                                         int64_t count, const double* __restrict__ wsums) {
  __shared__ int s_f;
  if (threadIdx.x == 0) {
    int fx;
    frexpf(fixed_scale(wsums[2]), &fx);  // 2^F = 2^(fx - 1)
    s_f = fx - 1;
  }
  __syncthreads();
  const int F = s_f;
  const int64_t stride = gstride(), total = g2 ? 2 * count : count;
  constexpr int U = 4;  // loads in flight
  for (int64_t i0 = gtid(); i0 < total; i0 += U * stride) {
    unsigned long long v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = i0 + u * stride;
      if (i < total) v[u] = i < count ? g1[i] : g2[i - count];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = i0 + u * stride;
      if (i < total) {
        double* out = reinterpret_cast<double*>(i < count ? g1 + i : g2 + (i - count));
        *out = fixed_value((long long)v[u], F);
      }
    }
  }
}

cudaError_t launch_fixed_to_double(unsigned long long* g1, unsigned long long* g2, int64_t count, const double* wsums,
                                   cudaStream_t s) {
  const int64_t blocks = std::min<int64_t>(num_sms() * 8, ((g2 ? 2 : 1) * count + 1023) / 1024);
  k_fixed_to_double<<<int(std::max<int64_t>(1, blocks)), 256, 0, s>>>(g1, g2, count, wsums); count_launch();
  return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_weight_sums(const float* __restrict__ w, int64_t n, double* __restrict__ sums) {
  double a = 0.0, b = 0.0, c = 0.0;
  for (int64_t i = gtid(); i < n; i += gstride()) {
    const double v = w[i];
    a += v;
    b += v * v;
    c += fabs(v);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
    c += __shfl_down_sync(0xffffffffu, c, o);
  }
  // one atomic per block and sum: the additions to one address queue up (three per warp took 47 us whatever n)
  __shared__ double red[3][8];
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = a;
    red[1][threadIdx.x >> 5] = b;
    red[2][threadIdx.x >> 5] = c;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double t = 0.0;
    for (int q = 0; q < 8; ++q) t += red[threadIdx.x][q];
    atomicAdd(sums + threadIdx.x, t);
  }
}

__global__ void k_set_sums(double* sums, double s1, double s2) {
  sums[0] = s1;
  sums[1] = s2;
  sums[2] = s1;
}

cudaError_t launch_weight_sums(const float* w, int64_t n, double* sums, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(sums, 0, 3 * sizeof(double), s);
  if (e != cudaSuccess || n == 0) return e;
  k_weight_sums<<<int(std::min<int64_t>(num_sms() * 4, (n + 1023) / 1024)), 256, 0, s>>>(w, n, sums); count_launch();
  return cudaGetLastError();
}

cudaError_t launch_set_sums(double* sums, double s1, double s2, cudaStream_t s) {
  k_set_sums<<<1, 1, 0, s>>>(sums, s1, s2); count_launch();
  return cudaGetLastError();
}

template <typename T>
__global__ void k_copy_rows(const T* __restrict__ src, int src_ld, T* __restrict__ dst, int dst_ld, int ng, int64_t rows) {
  const int64_t total = rows * ng;
  for (int64_t i = gtid(); i < total; i += gstride()) {
    const int64_t r = i / ng;
    const int z = int(i - r * ng);
    dst[r * dst_ld + z] = src[r * src_ld + z];
  }
}

template <typename T>
cudaError_t launch_copy_rows(const T* src, int src_ld, T* dst, int dst_ld, int ng, int64_t rows, cudaStream_t s) {
  k_copy_rows<T><<<num_sms() * 8, 256, 0, s>>>(src, src_ld, dst, dst_ld, ng, rows); count_launch();
  return cudaGetLastError();
}
template cudaError_t launch_copy_rows<float>(const float*, int, float*, int, int, int64_t, cudaStream_t);
template cudaError_t launch_copy_rows<double>(const double*, int, double*, int, int, int64_t, cudaStream_t);

}  // namespace pk
